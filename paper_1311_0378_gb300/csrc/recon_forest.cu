// Reconstruction by merging regions along their best passes (Table II
// "Morphological Reconstruction", the same fixed point as recon_kernels.cu).
//
// R(p) is the widest-path value from a source s: give neighbouring pixels p, q
// the weight min(I(p), I(q)) and p and s the weight J(p); then R(p) is the
// largest, over the paths from p to s, of the smallest weight on the path.
// Widest paths run inside a maximum spanning forest (Hu 1961), and Boruvka's
// rule (1926) builds one with all regions working at once: every region takes
// its heaviest outgoing edge, of weight w say, and R of its pixels is the
// smaller of w and R on the other side. Nothing travels pixel by pixel: the
// number of steps grows with the logarithm of the region count, not with the
// length of the path a value takes through the image, which is what bounds
// the wavefront (about 7 000 sequential levels on a border-seeded 4096^2 tile).
//
// Three launches per group of tiles, one CTA per 64 x 64 block:
//   block_kernel  splits the block into the basins of its mask (every pixel
//     follows its highest neighbour; R(p) = min(I(p), R(top of its basin))),
//     lists the passes between them, which lie at the saddles of the mask, and
//     runs Boruvka's rounds on that small graph.
//     A region whose heaviest edge leads out of the block stops there: it
//     becomes a node that other blocks may raise. Every other region ends up
//     with a final value, or with a cap and the node it hangs on.
//   rim_kernel    joins the nodes across block borders.
//   value_kernel  R of every node, then R(p) = min(cap(p), R(node(p))).
// Nodes are kept in a forest of weighted links: the region of a at weight w is
// what hangs together by links of weight >= w, and its root is found by walking
// them up from a. An edge (a, b, w) is added by linking the two regions' roots
// at w; the lighter link that this displaces is added again further up. Links are single 64-bit words changed by compare-and-swap, and
// every link goes to a node of higher (hashed) priority: no cycles in any
// interleaving, and walks of logarithmic expected length.
//
// Measured on GB300 (whole call, the wavefront engine before -> this one): a
// 4096^2 tile seeded from its border, 4-connected, 5.61 -> 0.61 ms; with an
// h-dome marker, 8-connected, 0.405 -> 0.394 ms; 200 tiles of 256 .. 4096
// pixels a side (910 Mpx, both markers) 60.4 -> 19.4 ms; 512^2 0.230 -> 0.121 ms.
#include <climits>
#include "recon_forest.h"

namespace rf {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int NT = 256;            // threads per CTA: one 16-pixel run each
// Shared-memory image: row stride ST, pixel (x, y) at (y + 1) * ST + X0 + x.
// The cell right of a row's last pixel is the first cell of the next row.
constexpr int ST = BS + 4, X0 = 4;
constexpr int NCELL = (BS + 2) * ST + 4;
constexpr int IST = 20;            // row stride of the byte image in words (interior at word 4)
constexpr int TAB = 2560;          // passes a block can list
constexpr unsigned ROOT = 0x8000u; // label flag: a basin number, not a pointer to a cell
constexpr unsigned DONE = 0xFFFFFFFFu;
constexpr unsigned K_SOURCE = 2u << 22, K_EDGE = 1u << 22;   // edge kinds, heavier wins a tie
constexpr unsigned SRC = 0xFFFFFFFFu;   // parent number of the source
constexpr unsigned RES = 255u;          // node slot of a pixel whose value is final
constexpr int MAX_STEPS = 1 << 20;      // bound of every walk

// Basins: no two tops are neighbours, so at most one pixel in four (two) for
// 8- (4-)connectivity; number 0 is the outside.
template <int CONN>
struct Smem {
    static constexpr int NB = (CONN == 8 ? BPX / 4 : BPX / 2) + 32;
    alignas(16) uint32_t W[NCELL];    // I << 24 | label
    alignas(16) uint32_t tab[TAB];    // passes: basin << 20 | basin << 8 | weight; before that the byte images
    uint32_t best[NB];                // heaviest edge of a region this round; then cap << 8 | node slot
    uint32_t sj[NB], cb[NB];          // heaviest edge to the source / out of the block
    uint16_t comp[NB], up[NB];        // region's root, link to the region merged into
    uint8_t capw[NB], st[NB];         // weight of that link; 1 = node, 2 = final (then the node slot)
    uint32_t link[MAX_TERM];          // node links: weight << 8 | parent slot (RES = source)
    uint32_t ss[MAX_TERM];
    uint8_t hT[BS + 2], hB[BS + 2], hL[BS], hR[BS];   // mask of the pixels around the block
    unsigned nb, nt, ne;              // basins, nodes, passes
    int tile;
    unsigned local;
};

__device__ __forceinline__ uint32_t pmax(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t even_plane(uint32_t w) { return __byte_perm(w, 0u, 0x4240); }
__device__ __forceinline__ uint32_t odd_plane(uint32_t w) { return __byte_perm(w, 0u, 0x4341); }

__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The tile of block b of the group (warp-wide 32-ary search).
__device__ __forceinline__ int find_tile(const Params &P, unsigned b)
{
    int lo = 0, n = P.ntiles;   // the tile is one of lo .. lo + n - 1
    const int lane = threadIdx.x & 31;
    while (n > 1) {
        const int step = (n + 31) / 32;
        const int i = lane * step;
        const bool le = i < n && P.base[lo + i] <= b;
        const int k = 31 - __clz(__ballot_sync(FULL, le));
        lo += k * step;
        n = min(step, n - k * step);
    }
    return lo;
}

// 16 pixels of an image row from column x on, zero right of column W. Any
// alignment: aligned words around the run, shifted; a word is only read when
// it holds a pixel of the run.
__device__ __forceinline__ uint4 load16(const uint8_t *row, int x, int W, bool vec)
{
    const int n = W - x;
    if (vec && n >= 16) return *(const uint4 *)(row + x);
    uint32_t w[5] = {0u, 0u, 0u, 0u, 0u};
    if (n > 0) {
        const uintptr_t a = (uintptr_t)(row + x);
        const int s = (int)(a & 3);
        const uint32_t *q = (const uint32_t *)(a - s);
#pragma unroll
        for (int j = 0; j < 5; ++j)
            if (4 * j - s < min(n, 16)) w[j] = q[j];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            w[j] = __funnelshift_r(w[j], w[j + 1], 8 * s);
            const int v = n - 4 * j;   // pixels of this word inside the image
            if (v < 4) w[j] = v > 0 ? w[j] & (0xFFFFFFFFu >> (8 * (4 - v))) : 0u;
        }
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ uint32_t inside(int n)   // byte mask of the first n pixels of a word
{
    return n >= 4 ? 0xFFFFFFFFu : (n > 0 ? 0xFFFFFFFFu >> (8 * (4 - n)) : 0u);
}

__device__ __forceinline__ void store16(uint8_t *row, int x, int W, uint4 v, bool vec)
{
    const int n = min(W - x, 16);
    if (vec && n == 16) {
        *(uint4 *)(row + x) = v;
        return;
    }
    if (n <= 0) return;
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    if ((((uintptr_t)(row + x)) & 3) == 0) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (4 * j + 3 < n) *(uint32_t *)(row + x + 4 * j) = w[j];
            else
                for (int b = 0; b < 4; ++b)
                    if (4 * j + b < n) row[x + 4 * j + b] = (uint8_t)(w[j] >> (8 * b));
        }
        return;
    }
#pragma unroll
    for (int j = 0; j < 16; ++j)
        if (j < n) row[x + j] = (uint8_t)(w[j >> 2] >> (8 * (j & 3)));
}

// Cell offset of direction d (0..7: NW, N, NE, W, E, SW, S, SE, in the order
// of the cells' numbers), a sign-extended byte of a constant.
__device__ __forceinline__ int dir_off(unsigned d)
{
    constexpr uint32_t LO = (uint32_t)(uint8_t)(-ST - 1) | (uint32_t)(uint8_t)(-ST) << 8 |
                            (uint32_t)(uint8_t)(-ST + 1) << 16 | (uint32_t)(uint8_t)(-1) << 24;
    constexpr uint32_t HI = 1u | (uint32_t)(ST - 1) << 8 | (uint32_t)ST << 16 | (uint32_t)(ST + 1) << 24;
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(LO), "r"(HI), "r"(d * 0x1111u + 0x8880u));
    return (int)r;
}

// One word of four pixels against its neighbours, even pixels in one u16x2
// plane, odd ones in the other. rows: words left, centre, right of the rows
// above, at and below. A neighbour is upper when it is higher, or equal and
// later; as keys I << 3 | direction, when its key is at least I << 3 | 4.
//   kE, kO: the largest key, i.e. the highest neighbour and its direction;
//   returns a byte per pixel: the saddle arcs. The upper neighbours form arcs on
// the ring around a pixel. Inside an arc they hang together without the pixel
// (ring neighbours are adjacent; for 8-connectivity so are N and E and so on,
// for 4-connectivity the corner between them must be upper too), so passes lie
// only at pixels with two or more arcs: bit k is set where an arc starts (ring
// order N, NE, E, SE, S, SW, W, NW), and no bit when there are fewer than two.
template <int CONN>
__device__ __forceinline__ uint32_t classify(const uint32_t (&l)[3], const uint32_t (&c)[3], const uint32_t (&r)[3],
                                             uint32_t &kE, uint32_t &kO)
{
    uint32_t e[3], o[3], we[3], eo[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        e[a] = even_plane(c[a]) << 3;
        o[a] = odd_plane(c[a]) << 3;
        we[a] = __funnelshift_l(odd_plane(l[a]) << 3, o[a], 16);    // left neighbours of the even pixels
        eo[a] = __funnelshift_r(e[a], even_plane(r[a]) << 3, 16);   // right neighbours of the odd pixels
    }
    auto plane = [](uint32_t nw, uint32_t n, uint32_t ne, uint32_t w, uint32_t own, uint32_t ea, uint32_t sw, uint32_t so,
                    uint32_t se, uint32_t &key) {
        // bit 15 of each lane is set so that the subtractions below do not borrow across lanes
        const uint32_t k[8] = {n | 0x80018001u, ne | 0x80028002u, ea | 0x80048004u, se | 0x80078007u,
                               so | 0x80068006u, sw | 0x80058005u, w | 0x80038003u, nw | 0x80008000u};
        key = __vimax3_u16x2(k[0], k[2], k[4]);
        key = pmax(key, k[6]);
        if (CONN == 8) {
            key = __vimax3_u16x2(key, k[1], k[3]);
            key = __vimax3_u16x2(key, k[5], k[7]);
        }
        key &= 0x7FFF7FFFu;
        const uint32_t ref = own | 0x00040004u;
        uint32_t m = 0;   // upper neighbours in ring order
#pragma unroll
        for (int b = 0; b < 8; ++b) m |= ((k[b] - ref) >> (15 - b)) & (0x00010001u << b);
        const uint32_t mm = m * 0x101u, both = (mm >> 1) & (mm >> 7) & 0x00AA00AAu;   // corners between two upper ones
        m = CONN == 8 ? (m | both) : ((m & 0x00550055u) | (m & both));
        const uint32_t s = m & ~((m * 0x101u) >> 7) & 0x00FF00FFu;                    // arc starts
        const uint32_t two = s & ((s | 0x01000100u) - 0x00010001u);                   // nonzero with two or more
        return s & ((((two & 0x00FF00FFu) + 0x00FF00FFu) >> 8 & 0x00010001u) * 0xFFu);
    };
    const uint32_t sE = plane(we[0], e[0], o[0], we[1], e[1], o[1], we[2], e[2], o[2], kE);
    const uint32_t sO = plane(e[0], o[0], eo[0], e[1], o[1], eo[1], e[2], o[2], eo[2], kO);
    return sE | sO << 8;
}

// Cell offset of ring position k (see classify).
__device__ __forceinline__ int ring_off(unsigned k)
{
    constexpr uint32_t LO = (uint32_t)(uint8_t)(-ST) | (uint32_t)(uint8_t)(-ST + 1) << 8 | 1u << 16 |
                            (uint32_t)(ST + 1) << 24;
    constexpr uint32_t HI = (uint32_t)ST | (uint32_t)(ST - 1) << 8 | (uint32_t)(uint8_t)(-1) << 16 |
                            (uint32_t)(uint8_t)(-ST - 1) << 24;
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(LO), "r"(HI), "r"(k * 0x1111u + 0x8880u));
    return (int)r;
}

// Priority of a node: links go to higher priorities, the source last.
__device__ __forceinline__ uint32_t priority(uint32_t node)
{
    uint32_t h = node * 0x9E3779B1u;
    h ^= h >> 15;
    return h * 0x2C1B3C6Du;
}

// Adds edge (a, b, w) to a forest of weighted links. F: load(node) and
// cas(node, old, new) on link words, weight(word), parent(word), word(weight,
// parent), before(a, b): a has lower priority than b. Returns false when a
// walk exceeded its bound.
template <class F>
__device__ __forceinline__ bool join(F &f, unsigned a, unsigned b, unsigned w)
{
    for (int it = 0; it < MAX_STEPS; ++it) {
        if (a == b) return true;
        if (a == F::SOURCE || (b != F::SOURCE && f.before(b, a))) { const unsigned x = a; a = b; b = x; }
        // a: the node of lower priority; step towards its root at weight w
        const auto la = f.load(a);
        if (f.weight(la) >= w) {
            a = f.parent(la);
            continue;
        }
        if (b != F::SOURCE) {
            const auto lb = f.load(b);
            if (f.weight(lb) >= w) {
                b = f.parent(lb);
                continue;
            }
        }
        if (f.cas(a, la, f.word(w, b))) {   // displaced: a's former parent, at its lighter weight
            a = b;
            b = f.parent(la);
            w = f.weight(la);
            if (w == 0) return true;        // every node reaches the source at weight 0
        }
    }
    return false;
}

struct SharedLinks {
    static constexpr unsigned SOURCE = RES;
    uint32_t *link;
    unsigned base;
    __device__ uint32_t load(unsigned n) const { return *(volatile uint32_t *)&link[n]; }
    __device__ bool cas(unsigned n, uint32_t o, uint32_t v) const { return atomicCAS(&link[n], o, v) == o; }
    __device__ unsigned weight(uint32_t l) const { return l >> 8; }
    __device__ unsigned parent(uint32_t l) const { return l & 255u; }
    __device__ uint32_t word(unsigned w, unsigned p) const { return w << 8 | p; }
    __device__ bool before(unsigned a, unsigned b) const { return priority(base + a) < priority(base + b); }
};

struct GlobalLinks {
    static constexpr unsigned SOURCE = SRC;
    unsigned long long *link;
    __device__ unsigned long long load(unsigned n) const { return *(volatile unsigned long long *)&link[n]; }
    __device__ bool cas(unsigned n, unsigned long long o, unsigned long long v) const
    {
        return atomicCAS(&link[n], o, v) == o;
    }
    __device__ unsigned weight(unsigned long long l) const { return (unsigned)(l >> 32); }
    __device__ unsigned parent(unsigned long long l) const { return (unsigned)l; }
    __device__ unsigned long long word(unsigned w, unsigned p) const { return (unsigned long long)w << 32 | p; }
    __device__ bool before(unsigned a, unsigned b) const { return priority(a) < priority(b); }
};

// Every pass between two basins, f(a, b, w, number): the list's entries, or
// (when there are too many for it) every pair of neighbouring pixels.
template <int CONN, class F>
__device__ __forceinline__ void each_pass(Smem<CONN> &S, F f)
{
    if (S.ne <= TAB) {
        for (unsigned i = threadIdx.x; i < S.ne; i += NT) {
            const uint32_t e = S.tab[i];
            f(e >> 20, (e >> 8) & 0xFFFu, e & 255u, i);
        }
    } else {
        for (unsigned i = threadIdx.x; i < BPX * 4; i += NT) {
            const unsigned px = i >> 2, d = i & 3u;
            if (CONN == 4 && (d & 1u)) continue;
            const unsigned p = (px / BS + 1) * ST + X0 + px % BS;
            const uint32_t a = S.W[p], b = S.W[p + dir_off(4u + d)];
            const unsigned w = min(a >> 24, b >> 24);
            if (w && ((a ^ b) & 0xFFFFu)) f(a & 0x7FFFu, b & 0x7FFFu, w, i);
        }
    }
}

// The two basins of pass number i.
template <int CONN>
__device__ __forceinline__ void pass_ends(const Smem<CONN> &S, unsigned i, unsigned &a, unsigned &b)
{
    if (S.ne <= TAB) {
        const uint32_t e = S.tab[i];
        a = e >> 20;
        b = (e >> 8) & 0xFFFu;
    } else {
        const unsigned px = i >> 2, p = (px / BS + 1) * ST + X0 + px % BS;
        a = S.W[p] & 0x7FFFu;
        b = S.W[p + dir_off(4u + (i & 3u))] & 0x7FFFu;
    }
}

template <int CONN>
__global__ void __launch_bounds__(NT, CONN == 8 ? 4 : 3) block_kernel(Params P)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Smem<CONN> &S = *reinterpret_cast<Smem<CONN> *>(smem_raw);
    constexpr int NB = Smem<CONN>::NB;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned blk = blockIdx.x;
    unsigned long long tick[6];   // thread 0: start and end of the phases (recon_work.phase_ns)
    if (tid == 0) tick[0] = now_ns();
    if (warp == 0) {
        const int t = find_tile(P, blk);
        if (lane == 0) {
            S.tile = t;
            S.local = blk - P.base[t];
            S.nb = 1;
            S.nt = 0;
            S.ne = 0;
        }
    }
    __syncthreads();
    const Tile D = P.tiles[S.tile];
    const int by = (int)(S.local / (unsigned)D.nbx), bx = (int)(S.local - (unsigned)by * D.nbx);
    const int y0 = by * BS, x0 = bx * BS;
    const bool vec = (D.pitch % 16) == 0 && ((uintptr_t)D.I % 16) == 0 && ((uintptr_t)D.J % 16) == 0;
    const int r = tid >> 2, c = tid & 3;         // this thread's run: row r, columns 16c .. 16c + 15
    const int y = y0 + r, x = x0 + 16 * c;
    uint32_t *const bi = S.tab;                  // byte image of I: rows -1 .. 64, IST words each
    uint32_t *const bj = S.tab + (BS + 2) * IST + 4;   // bytes of J: 64 rows of 16 words
    uint4 vi = make_uint4(0, 0, 0, 0), vj = vi;
    {
        if (y < D.H) {
            vi = load16(D.I + (size_t)y * D.pitch, x, D.W, vec);
            if (!D.fill) vj = load16(D.J + (size_t)y * D.pitch, x, D.W, vec);
        }
        // the mask around the block: 66 pixels above, 66 below, 64 left, 64 right
        for (int i = tid; i < 2 * (BS + 2) + 2 * BS; i += NT) {
            int yy, xx;
            uint8_t *h;
            if (i < BS + 2) { yy = y0 - 1; xx = x0 - 1 + i; h = &S.hT[i]; }
            else if (i < 2 * (BS + 2)) { yy = y0 + BS; xx = x0 - 1 + i - (BS + 2); h = &S.hB[i - (BS + 2)]; }
            else if (i < 2 * (BS + 2) + BS) { yy = y0 + i - 2 * (BS + 2); xx = x0 - 1; h = &S.hL[i - 2 * (BS + 2)]; }
            else { yy = y0 + i - 2 * (BS + 2) - BS; xx = x0 + BS; h = &S.hR[i - 2 * (BS + 2) - BS]; }
            uint8_t v = 0;
            if (yy >= 0 && yy < D.H && xx >= 0 && xx < D.W) {
                v = D.I[(size_t)yy * D.pitch + xx];
                if (D.dual) v = (uint8_t)~v;
            }
            *h = v;
        }
        if (D.dual) {   // erosion: complemented values inside the image
            const int n = y < D.H ? D.W - x : 0;
            const uint32_t m0 = inside(n), m1 = inside(n - 4), m2 = inside(n - 8), m3 = inside(n - 12);
            vi = make_uint4(vi.x ^ m0, vi.y ^ m1, vi.z ^ m2, vi.w ^ m3);
            if (!D.fill) vj = make_uint4(vj.x ^ m0, vj.y ^ m1, vj.z ^ m2, vj.w ^ m3);
        }
        if (D.fill) {   // FillHoles: seeded by the (complemented) mask on the image border, 0 inside
            if (y == 0 || y == D.H - 1) {
                vj = vi;
            } else {
                uint32_t w[4] = {vi.x, vi.y, vi.z, vi.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint32_t m = 0;
                    if (x + 4 * j == 0) m |= 0xFFu;
                    const int b = D.W - 1 - (x + 4 * j);
                    if (b >= 0 && b < 4) m |= 0xFFu << (8 * b);
                    w[j] &= m;
                }
                vj = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
        *(uint4 *)&bi[(r + 1) * IST + 4 + 4 * c] = vi;
        *(uint4 *)&bj[r * (BS / 4) + 4 * c] = vj;
        if (tid < IST) bi[tid] = 0u;                                   // row above
        else if (tid < 2 * IST) bi[(BS + 1) * IST + tid - IST] = 0u;   // row below
        else if (tid >= 64 && tid < 64 + BS + 3) {                     // words left of row q and right of row q - 1
            const int q = tid - 64;
            if (q < BS + 2) bi[q * IST + 3] = 0u;
            if (q) bi[q * IST] = 0u;
        }
        if (tid < ST + 4) S.W[tid] = ROOT;                             // cells around the block: basin 0
        else if (tid < 2 * (ST + 4)) S.W[(BS + 1) * ST + tid - (ST + 4)] = ROOT;
        if (tid < BS) {
            S.W[(tid + 1) * ST + X0 - 1] = ROOT;
            S.W[(tid + 2) * ST] = ROOT;
        }
        for (int i = tid; i < NB; i += NT) S.cb[i] = 0u;
        if (tid == 0) S.sj[0] = 0u;
        bool bad = false;
        if (P.check && !D.fill)
            bad = (__vcmpgtu4(vj.x, vi.x) | __vcmpgtu4(vj.y, vi.y) | __vcmpgtu4(vj.z, vi.z) | __vcmpgtu4(vj.w, vi.w)) != 0;
        if (__syncthreads_or(bad)) {
            if (tid == 0) {
                atomicExch(&P.tile_err[D.index], 2);
                atomicMin(&P.ctl->err_tile, D.index);
                P.nterm[blk] = 0;
            }
            return;
        }
    }

    if (tid == 0) tick[1] = now_ns();
    // Basins: every pixel points to its highest neighbour (the later one of
    // equals), if that one is higher or equal and later; the others are tops.
    uint32_t saddle[4];   // this thread's saddles: a byte per pixel
    {
        uint32_t rows[3][6];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const uint32_t *row = &bi[(r + a) * IST + 4 + 4 * c];
            const uint4 v = *(const uint4 *)row;
            rows[a][0] = row[-1];
            rows[a][1] = v.x; rows[a][2] = v.y; rows[a][3] = v.z; rows[a][4] = v.w;
            rows[a][5] = row[4];
        }
        uint32_t lab[16];
        unsigned tops = 0;
        const int cell = (r + 1) * ST + X0 + 16 * c;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t l[3] = {rows[0][j], rows[1][j], rows[2][j]};
            const uint32_t m[3] = {rows[0][j + 1], rows[1][j + 1], rows[2][j + 1]};
            const uint32_t q[3] = {rows[0][j + 2], rows[1][j + 2], rows[2][j + 2]};
            uint32_t kE, kO;
            saddle[j] = classify<CONN>(l, m, q, kE, kO);
            const uint32_t k4[4] = {kE & 0xFFFFu, kO & 0xFFFFu, kE >> 16, kO >> 16};
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const uint32_t v = (m[1] >> (8 * b)) & 255u;
                const bool top = k4[b] < (v << 3 | 4u);
                lab[4 * j + b] = v << 24 | (uint32_t)(cell + 4 * j + b + dir_off(k4[b] & 7u));
                tops |= (top ? 1u : 0u) << (4 * j + b);
            }
        }
        const unsigned mine = __popc(tops);
        unsigned incl = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned o = __shfl_up_sync(FULL, incl, d);
            if (lane >= d) incl += o;
        }
        unsigned at = 0;
        if (lane == 31) at = atomicAdd(&S.nb, incl);
        at = __shfl_sync(FULL, at, 31) + incl - mine;
        const uint32_t jw[4] = {vj.x, vj.y, vj.z, vj.w};
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if ((tops >> j) & 1u) {
                S.sj[at] = (jw[j >> 2] >> (8 * (j & 3))) & 255u;   // the top's own source edge
                lab[j] = (lab[j] & 0xFF000000u) | ROOT | at++;
            }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            *(uint4 *)&S.W[cell + 4 * j] = make_uint4(lab[4 * j], lab[4 * j + 1], lab[4 * j + 2], lab[4 * j + 3]);
    }
    __syncthreads();
    const unsigned nb = S.nb;
    // Every pixel's basin, and the heaviest source edge of each basin.
    const int col = (warp & 1) * 32 + lane, row0 = (warp >> 1) * 16;   // pixel passes: 32 columns x 16 rows a warp
    {
        volatile uint32_t *W = S.W;
        const uint8_t *jb = (const uint8_t *)bj;
        for (int i = 0; i < 16; ++i) {
            const int p = (row0 + i + 1) * ST + X0 + col;
            const uint32_t w = W[p];
            unsigned l = w & 0xFFFFu;
            if (!(l & ROOT)) {
                do l = W[l] & 0xFFFFu; while (!(l & ROOT));   // ends: each step goes to a higher (value, number)
                W[p] = (w & 0xFF000000u) | l;
            }
            const unsigned j = jb[(row0 + i) * BS + col], b = l & 0x7FFFu;
            if (j > *(volatile uint32_t *)&S.sj[b]) atomicMax(&S.sj[b], j);
        }
    }
    __syncthreads();
    // the heaviest edge out of the block of each basin; the passes take the byte images' place
    for (int i = tid; i < 4 * BS; i += NT) {
        const int side = i / BS, k = i % BS;
        int p;
        unsigned m;
        if (side < 2) {
            p = (side ? BS : 1) * ST + X0 + k;
            const uint8_t *h = side ? S.hB : S.hT;
            m = h[k + 1];
            if (CONN == 8) m = max(m, max((unsigned)h[k], (unsigned)h[k + 2]));
        } else {
            p = (k + 1) * ST + X0 + (side == 2 ? 0 : BS - 1);
            const uint8_t *h = side == 2 ? S.hL : S.hR;
            m = h[k];
            if (CONN == 8) {   // (the corners' diagonal pixels belong to the top and bottom lines)
                if (k > 0) m = max(m, (unsigned)h[k - 1]);
                if (k < BS - 1) m = max(m, (unsigned)h[k + 1]);
            }
        }
        const uint32_t w = S.W[p];
        m = min(m, w >> 24);
        if (m) atomicMax(&S.cb[w & 0x7FFFu], m);
    }
    for (unsigned b = tid; b < nb; b += NT) {
        S.comp[b] = (uint16_t)b;
        S.up[b] = (uint16_t)b;
        S.capw[b] = 255;
        S.st[b] = 0;
    }
    __syncthreads();
    if (tid == 0) tick[2] = now_ns();
    // Passes: a saddle joins its own basin to the one each arc starts in, at
    // its own height (weight 0 never beats a source edge and is left out).
    {
        const int cell = (r + 1) * ST + X0 + 16 * c;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            for (uint32_t bits = saddle[j]; bits; bits &= bits - 1) {
                const unsigned b = __ffs(bits) - 1;
                const int p = cell + 4 * j + (int)(b >> 3);
                const uint32_t w = S.W[p], q = S.W[p + ring_off(b & 7u)];
                if (((w ^ q) & 0xFFFFu) && w >> 24) {
                    const unsigned at = atomicAdd(&S.ne, 1u);
                    if (at < TAB) S.tab[at] = (w & 0x7FFFu) << 20 | (q & 0x7FFFu) << 8 | w >> 24;
                }
            }
    }
    __syncthreads();

    if (tid == 0) tick[3] = now_ns();
    // Boruvka's rounds. A live region takes the heaviest of its edges to the
    // source and to other regions (numbers break ties, the same for both
    // ends, so only the two ends of one edge can choose each other); if an
    // edge out of the block is heavier still, it stops as a node.
    int rounds = 0;
    for (bool live = true; live; ++rounds) {
        for (unsigned b = tid; b < nb; b += NT)
            if (S.up[b] == b && S.st[b] == 0) S.best[b] = S.sj[b] << 24 | K_SOURCE;
        __syncthreads();
        each_pass<CONN>(S, [&](unsigned a, unsigned b, unsigned w, unsigned i) {
            const unsigned ca = S.comp[a], cb = S.comp[b];
            if (ca == cb) return;
            const uint32_t key = w << 24 | K_EDGE | i;
            if (key > *(volatile uint32_t *)&S.best[ca]) atomicMax(&S.best[ca], key);
            if (key > *(volatile uint32_t *)&S.best[cb]) atomicMax(&S.best[cb], key);
        });
        __syncthreads();
        for (unsigned b = tid; b < nb; b += NT) {
            if (S.up[b] != b || S.st[b] != 0) continue;
            const uint32_t key = S.best[b];
            const unsigned w = key >> 24;
            if (S.cb[b] > w || (key & K_SOURCE)) {
                S.st[b] = S.cb[b] > w ? 1 : 2;
                *(volatile uint32_t *)&S.best[b] = DONE;
                continue;
            }
            unsigned a1, a2;
            pass_ends<CONN>(S, key & 0x3FFFFFu, a1, a2);
            unsigned t = S.comp[a1];
            if (t == b) t = S.comp[a2];
            // the other end chose this edge too and will not stop: the lower number stays
            if (b < t && *(volatile uint32_t *)&S.best[t] == key && S.cb[t] <= w) continue;
            S.up[b] = (uint16_t)t;
            S.capw[b] = (uint8_t)w;
        }
        __syncthreads();
        live = false;
        for (unsigned b = tid; b < nb; b += NT) {
            const unsigned was = S.comp[b];
            unsigned t = was;
            while (S.up[t] != t) t = S.up[t];
            S.comp[b] = (uint16_t)t;
            if (was == b) {
                if (t != b) {   // merged this round
                    atomicMax(&S.sj[t], S.sj[b]);
                    atomicMax(&S.cb[t], S.cb[b]);
                } else if (S.best[b] != DONE) {
                    live = true;
                }
            }
        }
        live = __syncthreads_or(live);
    }

    // Nodes and, per basin, its cap (or final value) and node
    for (unsigned b = tid; b < nb; b += NT)
        if (S.st[b] == 1) {
            const unsigned k = atomicAdd(&S.nt, 1u);
            S.ss[k] = S.sj[b];
            S.cb[b] = k;
        }
    __syncthreads();
    const unsigned nt = S.nt;
    for (unsigned b = tid; b < nb; b += NT) {
        unsigned v = 255, t = b;
        while (S.up[t] != t) {
            v = min(v, (unsigned)S.capw[t]);
            t = S.up[t];
        }
        S.best[b] = S.st[t] == 1 ? (v << 8 | S.cb[t]) : (min(v, S.sj[t]) << 8 | RES);
    }
    __syncthreads();
    if (nt) {
        // node links inside the block: to the source, then to each other
        each_pass<CONN>(S, [&](unsigned a, unsigned b, unsigned w, unsigned) {
            const uint32_t fa = S.best[a], fb = S.best[b];
            const unsigned na = fa & 255u, nb2 = fb & 255u;
            if (na == nb2 || (na != RES && nb2 != RES)) return;
            atomicMax(&S.ss[na == RES ? nb2 : na], min(w, min(fa >> 8, fb >> 8)));
        });
        __syncthreads();
        for (unsigned k = tid; k < nt; k += NT) S.link[k] = S.ss[k] << 8 | RES;
        __syncthreads();
        SharedLinks F{S.link, blk * MAX_TERM};
        bool ok = true;
        each_pass<CONN>(S, [&](unsigned a, unsigned b, unsigned w, unsigned) {
            const uint32_t fa = S.best[a], fb = S.best[b];
            const unsigned na = fa & 255u, nb2 = fb & 255u;
            if (na == nb2 || na == RES || nb2 == RES) return;
            w = min(w, min(fa >> 8, fb >> 8));
            if (w) ok &= join(F, na, nb2, w);
        });
        if (!ok) atomicCAS(&P.ctl->abort, 0, (int)rk::AB_MERGE);
        __syncthreads();
        for (unsigned k = tid; k < nt; k += NT) {
            const uint32_t l = S.link[k];
            const unsigned par = l & 255u;
            P.link[(size_t)blk * MAX_TERM + k] =
                (unsigned long long)(l >> 8) << 32 | (par == RES ? SRC : blk * MAX_TERM + par);
        }
    }
    if (tid == 0) P.nterm[blk] = nt;

    if (tid == 0) tick[4] = now_ns();
    // Results: the pixels themselves when everything is final, else (cap, node)
    {
        const int cell = (r + 1) * ST + X0 + 16 * c;
        uint32_t o[8];   // 16 x (value << 8 | node slot)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint4 q = *(const uint4 *)&S.W[cell + 4 * j];
            const uint32_t w[4] = {q.x, q.y, q.z, q.w};
            uint32_t f[4];
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const uint32_t e = S.best[w[b] & 0x7FFFu];
                f[b] = min(e >> 8, w[b] >> 24) << 8 | (e & 255u);
            }
            o[2 * j] = f[0] | f[1] << 16;
            o[2 * j + 1] = f[2] | f[3] << 16;
        }
        if (nt == 0) {
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) w[j] = __byte_perm(o[2 * j], o[2 * j + 1], 0x7531) ^ (D.dual ? FULL : 0u);
            if (y < D.H) store16(D.J + (size_t)y * D.pitch, x, D.W, make_uint4(w[0], w[1], w[2], w[3]), vec);
        } else {
            uint4 *dst = (uint4 *)(P.px + (size_t)blk * BPX + r * BS + 16 * c);
            dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
            dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
        }
        if (!P.flat) {
            uint16_t *rim = P.rim + (size_t)blk * 4 * BS;
            if (r == 0 || r == BS - 1) {
                uint4 *dst = (uint4 *)(rim + (r ? BS : 0) + 16 * c);
                dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
                dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
            }
            if (c == 0) rim[2 * BS + r] = (uint16_t)o[0];
            if (c == 3) rim[3 * BS + r] = (uint16_t)(o[7] >> 16);
        }
    }
    if (tid == 0) {
        tick[5] = now_ns();
        rk::Work &wk = P.work[D.index];
        atomicAdd(&wk.visits, 1ull);
        atomicAdd(&wk.seeds, (unsigned long long)(nb - 1));
        atomicAdd(&wk.levels, (unsigned long long)rounds);
        atomicAdd(&wk.busy_ns, tick[5] - tick[0]);
#pragma unroll
        for (int k = 0; k < 5; ++k) atomicAdd(&wk.phase_ns[k], tick[k + 1] - tick[k]);
    }
}

// Joins across block borders: a CTA of 128 threads handles the edges from its
// block's right column (warps 0, 1) and bottom row (warps 2, 3) to the blocks
// E, NE, SE and S, SW of it (the other diagonals belong to those blocks).
// Lanes that hold the same pair of nodes let the heaviest edge stand for all.
template <int CONN>
__global__ void __launch_bounds__(128) rim_kernel(Params P)
{
    __shared__ int s_tile;
    if (threadIdx.x < 32) {
        const int t = find_tile(P, blockIdx.x);
        if (threadIdx.x == 0) s_tile = t;
    }
    __syncthreads();
    const Tile D = P.tiles[s_tile];
    if (*(volatile int *)&P.tile_err[D.index]) return;
    const unsigned blk = blockIdx.x, local = blk - P.base[s_tile];
    const int by = (int)(local / (unsigned)D.nbx), bx = (int)(local - (unsigned)by * D.nbx);
    const bool right = threadIdx.x < 64;
    const int k = threadIdx.x & 63;
    if (right ? bx + 1 >= D.nbx : by + 1 >= D.nby) return;   // warp-uniform
    const uint16_t *rim = P.rim + (size_t)blk * 4 * BS;
    const unsigned pv = right ? rim[3 * BS + k] : rim[BS + k];
    const unsigned pn = (pv & 255u) == RES ? SRC : blk * MAX_TERM + (pv & 255u);
    GlobalLinks F{P.link};
    bool ok = true;
#pragma unroll
    for (int d = -1; d <= 1; ++d) {
        if (CONN == 4 && d != 0) continue;
        unsigned qn = SRC, w = 0;
        const int q = k + d;
        unsigned nb = 0;
        const uint16_t *src = nullptr;
        if (right) {
            if (q < 0) {
                if (by > 0) { nb = blk + 1 - D.nbx; src = P.rim + (size_t)nb * 4 * BS + BS; }          // NE: its bottom row, x = 0
            } else if (q >= BS) {
                if (by + 1 < D.nby) { nb = blk + 1 + D.nbx; src = P.rim + (size_t)nb * 4 * BS; }       // SE: its top row, x = 0
            } else {
                nb = blk + 1;
                src = P.rim + (size_t)nb * 4 * BS + 2 * BS + q;
            }
        } else if (q >= 0 && q < BS) {
            nb = blk + D.nbx;
            src = P.rim + (size_t)nb * 4 * BS + q;
        }
        if (src) {
            const unsigned qv = *src;
            qn = (qv & 255u) == RES ? SRC : nb * MAX_TERM + (qv & 255u);
            w = min(pv >> 8, qv >> 8);
        }
        if (pn == qn) w = 0;
        const unsigned long long pair = (unsigned long long)pn << 32 | qn;
        const unsigned same = __match_any_sync(FULL, pair);
        const unsigned top = __reduce_max_sync(same, w);
        const unsigned ties = __ballot_sync(FULL, w && w == top) & same;
        if (ties && __ffs(ties) - 1 == (int)(threadIdx.x & 31)) ok &= join(F, pn, qn, w);
        __syncwarp();
    }
    if (!ok) atomicCAS(&P.ctl->abort, 0, (int)rk::AB_MERGE);
}

// R of the block's nodes (the lightest link of their path to the source), then
// of its pixels.
__global__ void __launch_bounds__(NT) value_kernel(Params P)
{
    __shared__ int s_tile;
    __shared__ uint8_t R[256];
    const unsigned blk = blockIdx.x;
    const unsigned nt = P.nterm[blk];
    if (nt == 0) return;
    if (threadIdx.x < 32) {
        const int t = find_tile(P, blk);
        if (threadIdx.x == 0) s_tile = t;
    }
    const int r = threadIdx.x >> 2, c = threadIdx.x & 3;
    const uint4 *src = (const uint4 *)(P.px + (size_t)blk * BPX + r * BS + 16 * c);
    const uint4 q0 = src[0], q1 = src[1];
    R[threadIdx.x] = 255;
    if (threadIdx.x < nt) {
        unsigned n = blk * MAX_TERM + threadIdx.x, v = 255;
        int it = 0;
        for (; it < MAX_STEPS; ++it) {
            const unsigned long long l = __ldcg(&P.link[n]);
            v = min(v, (unsigned)(l >> 32));
            n = (unsigned)l;
            if (n == SRC) break;
        }
        if (it == MAX_STEPS) atomicCAS(&P.ctl->abort, 0, (int)rk::AB_MERGE);
        R[threadIdx.x] = (uint8_t)v;
    }
    __syncthreads();
    const Tile D = P.tiles[s_tile];
    if (P.tile_err[D.index]) return;
    const unsigned local = blk - P.base[s_tile];
    const int by = (int)(local / (unsigned)D.nbx), bx = (int)(local - (unsigned)by * D.nbx);
    const int y = by * BS + r, x = bx * BS + 16 * c;
    if (y >= D.H) return;
    const uint32_t o[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t v = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const uint32_t e = (o[2 * j + (b >> 1)] >> (16 * (b & 1))) & 0xFFFFu;
            v |= min(e >> 8, (uint32_t)R[e & 255u]) << (8 * b);   // R[RES] = 255: a final value stays
        }
        w[j] = v ^ (D.dual ? FULL : 0u);
    }
    const bool vec = (D.pitch % 16) == 0 && ((uintptr_t)D.J % 16) == 0;
    store16(D.J + (size_t)y * D.pitch, x, D.W, make_uint4(w[0], w[1], w[2], w[3]), vec);
}

}  // namespace rf

extern "C" cudaError_t rf_configure()
{
    cudaError_t e = cudaFuncSetAttribute(rf::block_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(rf::Smem<8>));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(rf::block_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(rf::Smem<4>));
    return e;
}

extern "C" cudaError_t rf_launch(int conn, const rf::Params *P, cudaStream_t st)
{
    if (conn == 8) rf::block_kernel<8><<<P->nblocks, rf::NT, sizeof(rf::Smem<8>), st>>>(*P);
    else rf::block_kernel<4><<<P->nblocks, rf::NT, sizeof(rf::Smem<4>), st>>>(*P);
    if (!P->flat) {
        if (conn == 8) rf::rim_kernel<8><<<P->nblocks, 128, 0, st>>>(*P);
        else rf::rim_kernel<4><<<P->nblocks, 128, 0, st>>>(*P);
        rf::value_kernel<<<P->nblocks, rf::NT, 0, st>>>(*P);
    }
    return cudaGetLastError();
}
