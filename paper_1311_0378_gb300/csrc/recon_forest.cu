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
//   block_kernel  splits the block into basins of its mask (every pixel follows
//     a neighbour at least as high; R(p) = min(I(p), R(top of its basin))),
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
// at w; the lighter link that this displaces is added again further up. Links
// are single 64-bit words changed by compare-and-swap, and every link goes to a
// node of higher (hashed) priority: no cycles in any interleaving, and walks of
// logarithmic expected length.
//
// Measured on GB300 (whole call, the wavefront engine -> this one): a 4096^2
// tile seeded from its border, 4-connected, 6.04 -> 0.280 ms; with an h-dome
// marker, 8-connected, 0.403 -> 0.203 ms; 200 tiles of 256 .. 4096 pixels a
// side (910 Mpx, both markers) 57.0 -> 9.44 ms; 512^2 0.231 -> 0.066 ms.
// block_kernel takes most of it (0.195 of 0.235 ms of kernel time on the
// border-seeded tile) and is bound by instruction issue and the shared-memory
// pipe (about 65% and 55%; DRAM below 4%), so what counts is warp instructions
// a block, 25 200 (h-dome) to 35 000 (border): hence saddles instead of all pixel
// pairs, arcs and targets of four pixels at once in byte lanes, loops rolled to
// fit the instruction cache, and lists that stay dense.
#include <climits>
#include <cstddef>
#include "recon_check.h"
#include "recon_forest.h"

namespace rf {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int NT = 256;            // threads per CTA: one 16-pixel run each
// Shared-memory label image: row stride ST, pixel (x, y) at (y + 1) * ST + X0 + x.
// The cell right of a row's last pixel is the first cell of the next row.
constexpr int ST = BS + 8, X0 = 8;
constexpr int NCELL = (BS + 2) * ST + 8;
constexpr int IST = ST / 4;        // row stride of the byte image in words, interior at word 2: a pixel's
                                   // byte has the number of its cell
constexpr int JOFF = (BS + 2) * IST + 4, IMG = JOFF + BPX / 4;   // where J's bytes start, words in all
static_assert(X0 == 8 && ST == 72, "layout");
constexpr int TAB = 2048;          // passes a block can list (noise has about 1150)
constexpr unsigned ROOT = 0x8000u; // label flag: a basin number, not a place of a cell
constexpr unsigned FINAL = 0xFFFFFFFEu, NODE = 0xFFFFFFFFu;   // best[] of a region that stopped
// edge kinds of a region's heaviest edge (weight << 24 | kind | number): the larger wins a tie
constexpr unsigned K_SOURCE = 2u << 22, K_EDGE = 1u << 22, K_OUT = 0u;
constexpr unsigned SRC = 0xFFFFFFFFu;   // parent number of the source
constexpr unsigned RES = 255u;          // node slot of a pixel whose value is final
constexpr int MAX_STEPS = 1 << 20;      // bound of every walk

// Basins: no two tops are neighbours, so at most one pixel in four (two) for
// 8- (4-)connectivity; number 0 is the outside.
template <int CONN>
struct Smem {
    static constexpr int NB = (CONN == 8 ? BPX / 4 : BPX / 2) + 32;
    alignas(16) uint16_t L[NCELL];    // labels: a cell's place in bytes, or ROOT | basin
    alignas(16) uint32_t img[IMG];    // byte image of I, then the bytes of J
    uint32_t tab[TAB];                // passes: region << 20 | region << 8 | weight, 0 = none
    uint32_t best[NB];                // heaviest edge of a live region to a region or out of the block; FINAL, NODE
    uint32_t sv[NB];                  // its heaviest source edge
    uint16_t comp[NB], up[NB];        // region's root (at the end cap << 8 | node slot), link to the region merged into
    uint8_t capw[NB];                 // weight of the up link; a final root's value; a node root's slot
    uint32_t link[MAX_TERM];          // node links: weight << 8 | parent slot (RES = source)
    uint8_t hT[BS + 2], hB[BS + 2], hL[BS], hR[BS];   // mask of the pixels around the block
    unsigned nb, nt, ne, nj;          // basins, nodes, passes, passes between nodes
    unsigned nlive[2];                // live roots, by round parity
    int tile;
    unsigned local;
    Block rec;                        // what is left for the other kernels
    unsigned long long tick[6];
};

__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The next kernel of a group may be launched while this one still runs (its
// CTAs fill the places that the last CTAs leave free); it waits for all of this
// one's results before it reads any: 4 us of a call on 512^2, 1% of the 910 Mpx
// batch's kernel time.
__device__ __forceinline__ void allow_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ const Tile &tile_of(const Params &P, int t) { return P.tiles ? P.tiles[t] : P.one; }

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

// 16 pixels of an image row from column x on, zero right of column W (n = W - x
// pixels are inside). Any alignment: aligned words around the run, shifted; a
// word is only read when it holds a pixel of the run.
__device__ __noinline__ uint4 load16_any(const uint8_t *at, int n)
{
    uint32_t w[5] = {0u, 0u, 0u, 0u, 0u};
    if (n > 0) {
        const int s = (int)((uintptr_t)at & 3);
        const uint32_t *q = (const uint32_t *)(at - s);
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

__device__ __forceinline__ uint4 load16(const uint8_t *at, int n, bool vec)
{
    if (vec && n >= 16) return *(const uint4 *)at;
    return load16_any(at, n);
}

__device__ __forceinline__ uint32_t inside(int n)   // byte mask of the first n pixels of a word
{
    return n >= 4 ? 0xFFFFFFFFu : (n > 0 ? 0xFFFFFFFFu >> (8 * (4 - n)) : 0u);
}

// The first n of 16 pixels to any address: whole words inside, bytes at the ends.
__device__ __noinline__ void store16_any(uint8_t *at, int n, uint4 v)
{
    n = min(n, 16);
    const int lead = (int)(-(intptr_t)at & 3);   // bytes before the first aligned word
    const uint32_t w[5] = {v.x, v.y, v.z, v.w, 0u};
    if (lead < n)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (lead + 4 * j + 4 <= n) *(uint32_t *)(at + lead + 4 * j) = __funnelshift_r(w[j], w[j + 1], 8 * lead);
    const int done = lead < n ? lead + (n - lead) / 4 * 4 : 0;   // words cover lead .. done - 1
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
        if (lead < n && i == lead) i = done;
        if (i >= n) break;
        const uint32_t q = i < 8 ? (i < 4 ? v.x : v.y) : (i < 12 ? v.z : v.w);
        at[i] = (uint8_t)(q >> (8 * (i & 3)));
    }
}

__device__ __forceinline__ void store16(uint8_t *at, int n, uint4 v, bool vec)
{
    if (vec && n >= 16) *(uint4 *)at = v;
    else if (n > 0) store16_any(at, n, v);
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

// One word of four pixels (bytes) against its neighbours. rows: words left,
// centre, right of the rows above, at and below. A neighbour is upper when it is
// higher, or equal and later in the image. The upper neighbours form arcs on the
// ring around a pixel (order N, NE, E, SE, S, SW, W, NW). Inside an arc they hang
// together without the pixel: ring neighbours are adjacent; for 8-connectivity so
// are N and E and so on, for 4-connectivity the corner between them must be upper
// too. Returns a byte per pixel with bit k set where an arc starts; bit 0 (N) when
// the ring is one closed arc; no bit when there is no upper neighbour.
template <int CONN>
__device__ __forceinline__ uint32_t arc_starts(const uint32_t (&l)[3], const uint32_t (&c)[3], const uint32_t (&r)[3])
{
    constexpr uint32_t H = 0x80808080u, ONES = 0x01010101u;
    const uint32_t own = c[1], ol = own & ~H, oh = own | H;
    uint32_t w[3], e[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        w[a] = __funnelshift_l(l[a], c[a], 8);   // left neighbours
        e[a] = __funnelshift_r(c[a], r[a], 8);   // right neighbours
    }
    // high bit of each byte: a later neighbour is at least as high / an earlier one is higher.
    // Bytes compare by their high bits, and where those agree by a subtraction of the low seven
    // bits below a guard bit.
    auto later = [&](uint32_t q) { const uint32_t t = (q | H) - ol; return (q & ~own) | (~(q ^ own) & t); };
    auto earlier = [&](uint32_t q) { const uint32_t t = oh - (q & ~H); return ~((own & ~q) | (~(own ^ q) & t)); };
    uint32_t m = (earlier(c[0]) >> 7) & ONES;
    m |= (earlier(e[0]) >> 6) & (ONES << 1);
    m |= (later(e[1]) >> 5) & (ONES << 2);
    m |= (later(e[2]) >> 4) & (ONES << 3);
    m |= (later(c[2]) >> 3) & (ONES << 4);
    m |= (later(w[2]) >> 2) & (ONES << 5);
    m |= (earlier(w[1]) >> 1) & (ONES << 6);
    m |= earlier(w[0]) & H;
    const uint32_t both = (((m >> 1) & 0x2A2A2A2Au) | ((m << 7) & H)) & (m << 1);   // corners (odd bits) between two upper ones
    m = CONN == 8 ? (m | both) : ((m & 0x55555555u) | (m & both));
    const uint32_t prev = ((m << 1) & 0xFEFEFEFEu) | ((m >> 7) & ONES);             // bit k: position k - 1 is upper
    const uint32_t closed = ((m & ~H) + ONES) & m & H;
    return (m & ~prev) | closed >> 7;
}

// High bit of each nonzero byte.
__device__ __forceinline__ uint32_t nonzero_bytes(uint32_t v) { return (((v & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | v) & 0x80808080u; }

// Cell offset of ring position k (see arc_starts).
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

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

// Cell offsets of four ring positions (bytes), plus RING0.
constexpr int RING0 = ST + 1;
__device__ __forceinline__ uint32_t ring_offs(uint32_t k)
{
    constexpr uint32_t LO = (uint32_t)(RING0 - ST) | (uint32_t)(RING0 - ST + 1) << 8 | (uint32_t)(RING0 + 1) << 16 |
                            (uint32_t)(RING0 + ST + 1) << 24;
    constexpr uint32_t HI = (uint32_t)(RING0 + ST) | (uint32_t)(RING0 + ST - 1) << 8 | (uint32_t)(RING0 - 1) << 16 |
                            (uint32_t)(RING0 - ST - 1) << 24;
    const uint32_t n = k | k >> 4;                    // positions 0 and 1 in byte 0, 2 and 3 in byte 2
    return prmt(LO, HI, prmt(n, 0u, 0x4420u));
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
        // both ends step towards their roots at weight w; the source is its own root
        const typename F::Word la = a == F::SOURCE ? 0 : f.load(a), lb = b == F::SOURCE ? 0 : f.load(b);
        const bool ua = a != F::SOURCE && f.weight(la) >= w, ub = b != F::SOURCE && f.weight(lb) >= w;
        if (ua) a = f.parent(la);
        if (ub) b = f.parent(lb);
        if (ua || ub) continue;
        // two roots: the one of lower priority is linked, and what that displaces (its former
        // parent, at a lighter weight) is added next
        const bool swap = a == F::SOURCE || (b != F::SOURCE && f.before(b, a));
        const unsigned lo = swap ? b : a, hi = swap ? a : b;
        const typename F::Word l = swap ? lb : la;
        if (f.cas(lo, l, f.word(w, hi))) {
            a = hi;
            b = f.parent(l);
            w = f.weight(l);
            if (w == 0) return true;        // every node reaches the source at weight 0
        } else {
            a = lo;
            b = hi;
        }
    }
    return false;
}

struct SharedLinks {
    typedef uint32_t Word;
    static constexpr unsigned SOURCE = RES;
    uint32_t *link;
    unsigned base;
    __device__ uint32_t load(unsigned n) const { return RK_CHECK(n < RES, CK_SLOT) ? *(volatile uint32_t *)&link[n] : (uint32_t)RES; }
    __device__ bool cas(unsigned n, uint32_t o, uint32_t v) const
    {
        return RK_CHECK(n < RES, CK_SLOT) ? atomicCAS(&link[n], o, v) == o : true;
    }
    __device__ unsigned weight(uint32_t l) const { return l >> 8; }
    __device__ unsigned parent(uint32_t l) const { return l & 255u; }
    __device__ uint32_t word(unsigned w, unsigned p) const { return w << 8 | p; }
    __device__ bool before(unsigned a, unsigned b) const { return priority(base + a) < priority(base + b); }
};

struct GlobalLinks {
    typedef unsigned long long Word;
    static constexpr unsigned SOURCE = SRC;
    unsigned long long *link;
    unsigned nodes;   // node numbers are below this
    __device__ unsigned long long load(unsigned n) const
    {
        return RK_CHECK(n < nodes, CK_NODE) ? *(volatile unsigned long long *)&link[n] : (unsigned long long)SRC;
    }
    __device__ bool cas(unsigned n, unsigned long long o, unsigned long long v) const
    {
        return RK_CHECK(n < nodes, CK_NODE) ? atomicCAS(&link[n], o, v) == o : true;
    }
    __device__ unsigned weight(unsigned long long l) const { return (unsigned)(l >> 32); }
    __device__ unsigned parent(unsigned long long l) const { return (unsigned)l; }
    __device__ unsigned long long word(unsigned w, unsigned p) const { return (unsigned long long)w << 32 | p; }
    __device__ bool before(unsigned a, unsigned b) const { return priority(a) < priority(b); }
};

// A block with more passes than its list holds works on every pair of
// neighbouring pixels instead: pair i is pixel i / 4 and its E, SW, S or SE
// neighbour.
template <int CONN, class F>
__device__ __noinline__ void each_pair(Smem<CONN> &S, F f)
{
    const uint8_t *img = (const uint8_t *)S.img;
    for (unsigned i = threadIdx.x; i < BPX * 4; i += NT) {
        const unsigned px = i >> 2, d = i & 3u;
        if (CONN == 4 && (d & 1u)) continue;
        const int py = (int)(px / BS), qx = (int)(px % BS);
        const int dx = d == 0 ? 1 : (int)d - 2, dy = d != 0;
        const unsigned a = S.L[(py + 1) * ST + X0 + qx], b = S.L[(py + dy + 1) * ST + X0 + qx + dx];
        const unsigned w = min(img[(py + 1) * ST + X0 + qx], img[(py + dy + 1) * ST + X0 + qx + dx]);
        if (w && a != b) f(a & 0x7FFFu, b & 0x7FFFu, w, i);
    }
}

// Five CTAs an SM where shared memory allows it (8-connectivity: 43 KB; 4: 56 KB
// for twice the basins), in 48 registers without spills, for which the timers and the
// tile's record are in shared memory: 5% of the 910 Mpx batch's kernel time against
// five CTAs with spills, 7% against four.
template <int CONN>
__global__ void __launch_bounds__(NT, CONN == 8 ? 5 : 4) block_kernel(const __grid_constant__ Params P)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Smem<CONN> &S = *reinterpret_cast<Smem<CONN> *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned blk = blockIdx.x;
    if (tid == 0) S.tick[0] = now_ns();   // start and end of the phases (recon_work.phase_ns)
    if (P.next && blk == 0 && tid < (int)(sizeof(Status) / 4))
        ((unsigned *)P.next)[tid] = tid == (int)(offsetof(rk::Ctl, err_tile) / 4) ? (unsigned)INT_MAX : 0u;
    if (warp == 0) {
        const int t = find_tile(P, blk);
        if (lane == 0) {
            S.tile = t;
            S.local = blk - (P.tiles ? P.base[t] : 0u);
            S.nb = 1;
            S.nt = 0;
            S.ne = 0;
            S.nj = 0;
            S.nlive[0] = S.nlive[1] = 0;
        }
    }
    __syncthreads();
    const Tile D = tile_of(P, S.tile);
    const int by = (int)(S.local / (unsigned)D.nbx), bx = (int)(S.local - (unsigned)by * D.nbx);
    const int y0 = by * BS, x0 = bx * BS;
    if (tid == 0)
        S.rec = Block{S.tile, S.local, D.nbx,
                      (bx + 1 < D.nbx ? B_RIGHT : 0u) | (by + 1 < D.nby ? B_DOWN : 0u) | (by > 0 ? B_UP : 0u)};
    const bool vec = (D.pitch % 16) == 0 && ((uintptr_t)D.I % 16) == 0 && ((uintptr_t)D.J % 16) == 0;
    const int r = tid >> 2, c = tid & 3;         // this thread's run: row r, columns 16c .. 16c + 15
    const int y = y0 + r, x = x0 + 16 * c;
    uint32_t *const bi = S.img;                  // I: rows -1 .. 64, IST words each, 0 around the block
    uint32_t *const bj = S.img + JOFF;           // J: 64 rows of 16 words
    {
        uint4 vi = make_uint4(0, 0, 0, 0), vj = vi;
        if (y < D.H) {
            vi = load16(D.I + (size_t)y * D.pitch + x, D.W - x, vec);
            if (!D.fill) vj = load16(D.J + (size_t)y * D.pitch + x, D.W - x, vec);
        }
        // the mask around the block: 66 pixels above, 66 below, 64 left, 64 right
        #pragma unroll 1
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
        *(uint2 *)&bi[(r + 1) * IST + 2 + 4 * c] = make_uint2(vi.x, vi.y);
        *(uint2 *)&bi[(r + 1) * IST + 4 + 4 * c] = make_uint2(vi.z, vi.w);
        if (tid < IST) bi[tid] = 0u;                                   // row above
        else if (tid < 2 * IST) bi[(BS + 1) * IST + tid - IST] = 0u;   // row below
        else if (tid >= 64 && tid < 64 + BS + 3) {                     // words left of row q and right of row q - 1
            const int q = tid - 64;
            if (q < BS + 2) bi[q * IST + 1] = 0u;
            if (q) bi[q * IST] = 0u;
        }
        *(uint4 *)&bj[r * (BS / 4) + 4 * c] = vj;
        if (tid < ST + 8) S.L[tid] = ROOT;                             // cells around the block: basin 0
        else if (tid < 2 * (ST + 8)) S.L[(BS + 1) * ST + tid - (ST + 8)] = ROOT;
        if (tid < BS) {
            S.L[(tid + 1) * ST + X0 - 1] = ROOT;
            S.L[(tid + 2) * ST] = ROOT;
        }
        if (tid == 0) { S.sv[0] = 0u; S.capw[0] = 0; }
        bool bad = false;
        if (P.check && !D.fill)
            bad = (__vcmpgtu4(vj.x, vi.x) | __vcmpgtu4(vj.y, vi.y) | __vcmpgtu4(vj.z, vi.z) | __vcmpgtu4(vj.w, vi.w)) != 0;
        if (__syncthreads_or(bad)) {
            if (tid == 0) {
                atomicExch(&P.tile_err[D.index], 2);
                atomicMin(&P.ctl->err_tile, D.index);
                P.block[blk] = Block{S.tile, S.local, D.nbx, 0u};
            }
            return;
        }
    }

    allow_next();
    if (tid == 0) S.tick[1] = now_ns();
    // Basins: every pixel points to the first upper neighbour of its first arc
    // (its heaviest edges all weigh its own height); pixels without one are tops.
    // A lane takes a word of four pixels in each of four rows: 4.5 loads and a
    // quarter of a warp's scan a word instead of the 9 and one that a row each
    // takes (8% of the 910 Mpx batch's kernel time).
    {
        constexpr int RL = BS / (NT / 16);
        const int row = RL * (2 * warp + (lane >> 4)), cw = lane & 15;
        const int cell = (row + 1) * ST + X0 + 4 * cw;
        uint32_t rest[RL], tops = 0u;    // further arcs; pixels without any (bit 8 b + 7 - row)
        unsigned passes = 0;
        {
            const uint32_t *at = &bi[(row + 1) * IST + 2 + cw];
            uint32_t l[3] = {0u, at[-IST - 1], at[-1]}, m[3] = {0u, at[-IST], at[0]}, q[3] = {0u, at[-IST + 1], at[1]};
#pragma unroll
            for (int h = 0; h < RL; ++h) {
#pragma unroll
                for (int k = 0; k < 2; ++k) { l[k] = l[k + 1]; m[k] = m[k + 1]; q[k] = q[k + 1]; }
                l[2] = at[(h + 1) * IST - 1]; m[2] = at[(h + 1) * IST]; q[2] = at[(h + 1) * IST + 1];
                const uint32_t high = nonzero_bytes(m[1]);   // pixels of height 0 have value 0, like the outside (basin 0)
                const uint32_t starts = arc_starts<CONN>(l, m, q) & ((high >> 7) * 255u);
                rest[h] = starts & ((starts | 0x80808080u) - 0x01010101u);   // without the lowest: further arcs
                const uint32_t some = nonzero_bytes(starts);
                tops |= (high & ~some) >> h;
                passes += __popc(rest[h]);
                // the targets' cells, as 16-bit lanes: ring position of the first arc (ones below its bit, counted
                // per byte), looked up for all four pixels at once
                uint32_t t = (starts & ~rest[h]) - (some >> 7);
                t -= (t >> 1) & 0x55555555u;
                t = (t & 0x33333333u) + ((t >> 2) & 0x33333333u);
                t = (t + (t >> 4)) & 0x0F0F0F0Fu;
                const uint32_t off = ring_offs(t);
                const uint32_t from = (unsigned)(cell + h * ST - RING0) * 0x10001u + 0x10000u;
                const uint32_t f0 = from + prmt(off, 0u, 0x4140u), f1 = from + 0x20002u + prmt(off, 0u, 0x4342u);
                const uint32_t m0 = prmt(some, 0u, 0x9988u), m1 = prmt(some, 0u, 0xBBAAu);
                *(uint2 *)&S.L[cell + h * ST] = make_uint2((2u * f0 & m0) | (ROOT * 0x10001u & ~m0), (2u * f1 & m1) | (ROOT * 0x10001u & ~m1));
            }
        }
        asm volatile("" ::: "memory");   // the tops' labels, of another type, come after
        // numbers for the tops (low half), places for the passes (high half)
        const unsigned mine = __popc(tops) | passes << 16;
        unsigned incl = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned o = __shfl_up_sync(FULL, incl, d);
            if (lane >= d) incl += o;
        }
        unsigned id = 0, slot = 0;
        if (lane == 31) {
            id = atomicAdd(&S.nb, incl & 0xFFFFu);
            slot = atomicAdd(&S.ne, incl >> 16);
        }
        id = __shfl_sync(FULL, id, 31) + ((incl - mine) & 0xFFFFu);
        slot = __shfl_sync(FULL, slot, 31) + ((incl - mine) >> 16);
        const uint8_t *const j0 = (const uint8_t *)&bj[row * (BS / 4) + cw];
#pragma unroll 1
        for (; tops; ++id) {
            const unsigned k = 31 - __clz(tops), b = k >> 3, h = ~k & 7u;
            tops ^= 1u << k;
            if (!RK_CHECK(id < (unsigned)Smem<CONN>::NB && cell + (int)(h * ST + b) < NCELL, CK_BASIN)) continue;
            S.L[cell + (int)(h * ST + b)] = (uint16_t)(ROOT | id);
            S.sv[id] = j0[h * BS + b];                       // the top's own source edge
        }
        // a pass lies at a pixel and leads to a further arc of it: cell << 3 | ring position
        const bool fits = slot + passes <= TAB;
#pragma unroll
        for (int h = 0; h < RL; ++h) {
#pragma unroll 1
            for (uint32_t bits = fits ? rest[h] : 0u; bits; ++slot) {
                const unsigned k = 31 - __clz(bits);
                bits ^= 1u << k;
                if (RK_CHECK(slot < (unsigned)TAB, CK_PASS)) S.tab[slot] = 8u * (unsigned)(cell + h * ST) + k;
            }
        }
    }
    __syncthreads();
    const unsigned nb = S.nb;
    // Every pixel's basin, and the heaviest source edge of each basin. A pixel
    // takes its target's label until that is a basin; all warps do so at once,
    // so paths halve as they are walked (each step goes to a higher (value,
    // number), so they end). 16 pixels a thread, their loads in flight together.
#pragma unroll 1
    for (unsigned b = tid; b < nb; b += NT) {
        S.best[b] = b ? 0u : FINAL;   // (the outside has value 0)
        S.up[b] = S.comp[b] = (uint16_t)b;
    }
    {
        const unsigned L = (unsigned)__cvta_generic_to_shared(S.L);
        auto label = [&](unsigned at) {
            if (!RK_CHECK(at < 2u * NCELL && !(at & 1u), CK_LABEL)) return ROOT;
            unsigned short v;
            asm volatile("ld.volatile.shared.u16 %0, [%1];" : "=h"(v) : "r"(L + at) : "memory");
            return (unsigned)v;
        };
        const int row0 = 2 * warp + (lane >> 4), cw = lane & 15;   // words as above: rows row0 + 16 i
        uint2 *const word = (uint2 *)&S.L[(row0 + 1) * ST + X0 + 4 * cw];
        constexpr int STEP = 16 * ST / 4;
        unsigned l[16];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint2 v = word[i * STEP];
            l[4 * i] = v.x & 0xFFFFu;
            l[4 * i + 1] = v.x >> 16;
            l[4 * i + 2] = v.y & 0xFFFFu;
            l[4 * i + 3] = v.y >> 16;
        }
        for (;;) {
            unsigned all = ROOT;
#pragma unroll
            for (int k = 0; k < 16; ++k) all &= l[k];
            if (all) break;
            unsigned n[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) n[k] = (l[k] & ROOT) ? l[k] : label(l[k]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                asm volatile("st.volatile.shared.v2.u32 [%0], {%1, %2};" :: "r"((unsigned)__cvta_generic_to_shared(&word[i * STEP])),
                             "r"(n[4 * i] | n[4 * i + 1] << 16), "r"(n[4 * i + 2] | n[4 * i + 3] << 16) : "memory");
            }
#pragma unroll
            for (int k = 0; k < 16; ++k) l[k] = n[k];
        }
        unsigned over = 0;   // pixels with a heavier source edge than their basin has so far
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t jw = bj[(row0 + 16 * i) * (BS / 4) + cw];
            if (jw == 0u) continue;
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if (RK_CHECK(l[4 * i + b] - ROOT < nb, CK_BASIN))
                    over |= (((jw >> (8 * b)) & 255u) > S.sv[l[4 * i + b] - ROOT] ? 1u : 0u) << (4 * i + b);
        }
#pragma unroll 1
        for (; over; over &= over - 1) {
            const int k = __ffs(over) - 1, i = k >> 2, row = row0 + 16 * i;
            const unsigned j = ((const uint8_t *)bj)[row * BS + 4 * cw + (k & 3)];
            atomicMax(&S.sv[S.L[(row + 1) * ST + X0 + 4 * cw + (k & 3)] - ROOT], j);
        }
    }
    __syncthreads();
    if (tid == 0) S.tick[2] = now_ns();
    // Maxima are taken without a look at the present one first: the load and the
    // compare cost more than the reductions they save (6% of the 910 Mpx batch's
    // kernel time).
    auto offer = [&](unsigned a, uint32_t key) {
        if (RK_CHECK(a < nb, CK_BASIN)) atomicMax(&S.best[a], key);
    };
    // Passes join a saddle's own basin to the one the arc starts in. A pass no
    // heavier than the source edges of both ends is never taken. The first
    // round's maxima are taken here too.
    const unsigned ne = S.ne;
    const bool listed = ne <= TAB;   // else: pairs of pixels instead of passes
    // Each warp has an eighth of the list to itself and keeps it dense: what a
    // pass (of the kernel over the list) drops is closed up, places only shrink.
    const unsigned seg0 = listed ? (ne * warp) / (NT / 32) : 0u;
    unsigned mine = listed ? (ne * (warp + 1)) / (NT / 32) - seg0 : 0u;   // the warp's passes
    auto close_up = [&](unsigned &to, uint32_t e) {   // keeps nonzero e; returns its place (warp-wide)
        const unsigned keep = __ballot_sync(FULL, e != 0u), at = to + __popc(keep & ((1u << lane) - 1u));
        if (e && RK_CHECK(at < (unsigned)TAB, CK_PASS)) S.tab[at] = e;
        to += __popc(keep);
        return at;
    };
    {
        unsigned to = seg0;
#pragma unroll 1
        for (unsigned k = 0; k < mine; k += 32) {
            uint32_t n = 0u;
            if (k + lane < mine &&
                RK_CHECK(seg0 + k + lane < (unsigned)TAB && S.tab[seg0 + k + lane] >> 3 < (unsigned)NCELL, CK_PASS)) {
                const uint32_t e = S.tab[seg0 + k + lane], p = e >> 3, w = ((const uint8_t *)bi)[p];
                const unsigned a = S.L[p] & 0x7FFFu, b = S.L[(int)p + ring_off(e & 7u)] & 0x7FFFu;
                if (RK_CHECK(a < nb && b < nb, CK_BASIN) && a != b && (w > S.sv[a] || w > S.sv[b])) n = a << 20 | b << 8 | w;
            }
            const unsigned at = close_up(to, n);
            if (n) {
                offer(n >> 20, n << 24 | K_EDGE | at);
                offer((n >> 8) & 0xFFFu, n << 24 | K_EDGE | at);
            }
        }
        mine = to - seg0;
    }
    // this thread's edge out of the block: pixel tid & 63 of side tid >> 6 (top, bottom, left, right)
    unsigned ob, ow;
    {
        const int side = tid >> 6, k = tid & 63;
        const int px = side < 2 ? k : (side == 2 ? 0 : BS - 1), py = side < 2 ? (side ? BS - 1 : 0) : k;
        const uint8_t *h = side < 2 ? (side ? S.hB : S.hT) + 1 : (side == 2 ? S.hL : S.hR);
        ow = h[k];
        if (CONN == 8) {   // (the corners' diagonal pixels belong to the top and bottom lines)
            if (side < 2 || k > 0) ow = max(ow, (unsigned)h[k - 1]);
            if (side < 2 || k < BS - 1) ow = max(ow, (unsigned)h[k + 1]);
        }
        ow = min(ow, (unsigned)((const uint8_t *)bi)[(py + 1) * ST + X0 + px]);
        ob = S.L[(py + 1) * ST + X0 + px] & 0x7FFFu;
        if (ow) offer(ob, ow << 24 | K_OUT);
    }
    __syncthreads();
    if (!listed) {
#pragma unroll 1
        for (unsigned b = 1 + tid; b < nb; b += NT) S.best[b] = 0u;
        __syncthreads();
    }

    if (tid == 0) S.tick[3] = now_ns();
    // Boruvka's rounds. A live region takes the heaviest of its edges: to the
    // source, to another region (numbers break ties, the same for both ends,
    // so only the two ends of one edge can choose each other) or out of the
    // block, where it stops as a node.
    // Live roots: in the first round all basins, then a list, which at least
    // halves with every round (a live root stops, merges or takes in another):
    // one of NB / 2 places for the odd rounds, one of NB / 4 for the even ones,
    // where the bytes of J were.
    uint16_t *const lists = (uint16_t *)bj;
    static_assert(Smem<CONN>::NB / 2 + Smem<CONN>::NB / 4 <= BPX / 2, "lists");
    unsigned nlive = nb - 1;
    int rounds = 0;
    for (;; ++rounds) {
        const uint16_t *now = lists + (rounds & 1 ? 0 : Smem<CONN>::NB / 2);
        uint16_t *next = lists + (rounds & 1 ? Smem<CONN>::NB / 2 : 0);
        // edges: to their present ends; one inside a region is dropped
        if (rounds || !listed) {
            if (tid == 0) S.nlive[rounds & 1] = 0;   // last read two rounds ago
            ob = S.comp[ob];
            if (ow) offer(ob, ow << 24 | K_OUT);
            if (listed) {
                unsigned to = seg0;
#pragma unroll 1
                for (unsigned k = 0; k < mine; k += 32) {
                    uint32_t n = 0u;
                    if (k + lane < mine && RK_CHECK(seg0 + k + lane < (unsigned)TAB, CK_PASS)) {
                        const uint32_t e = S.tab[seg0 + k + lane];
                        const unsigned a = S.comp[e >> 20], b = S.comp[(e >> 8) & 0xFFFu];
                        if (a != b) n = a << 20 | b << 8 | (e & 255u);
                    }
                    const unsigned at = close_up(to, n);
                    if (n) {
                        offer(n >> 20, n << 24 | K_EDGE | at);
                        offer((n >> 8) & 0xFFFu, n << 24 | K_EDGE | at);
                    }
                }
                mine = to - seg0;
            } else {
#pragma unroll 1
                for (unsigned b = 1 + tid; b < nb; b += NT) {   // all pixels' basins need their roots
                    unsigned t = b;
#pragma unroll 1
                    for (unsigned u; (u = S.up[t]) != t;) t = u;
                    S.comp[b] = (uint16_t)t;
                }
                __syncthreads();
                each_pair(S, [&](unsigned a, unsigned b, unsigned w, unsigned i) {
                    a = S.comp[a];
                    b = S.comp[b];
                    if (a == b) return;
                    offer(a, w << 24 | K_EDGE | i);
                    offer(b, w << 24 | K_EDGE | i);
                });
            }
            __syncthreads();
        }
#pragma unroll 1
        for (unsigned k = tid; k < nlive; k += NT) {
            const unsigned b = rounds ? now[k] : k + 1;
            if (!RK_CHECK(b < nb, CK_BASIN)) continue;
            const uint32_t key = S.best[b], src = S.sv[b] << 24 | K_SOURCE;
            if (src > key) {
                S.capw[b] = (uint8_t)(src >> 24);
                *(volatile uint32_t *)&S.best[b] = FINAL;
                continue;
            }
            if (!(key & K_EDGE)) {
                S.capw[b] = (uint8_t)atomicAdd(&S.nt, 1u);
                (void)RK_CHECK(S.capw[b] < RES, CK_SLOT);
                *(volatile uint32_t *)&S.best[b] = NODE;
                continue;
            }
            const unsigned i = key & 0x3FFFFFu;
            unsigned t, t2;
            if (listed) {
                if (!RK_CHECK(i < (unsigned)TAB, CK_PASS)) continue;
                const uint32_t e = S.tab[i];
                t = e >> 20;
                t2 = (e >> 8) & 0xFFFu;
            } else {
                const unsigned px = i >> 2, p = (px / BS + 1) * ST + X0 + px % BS;
                t = S.comp[S.L[p] & 0x7FFFu];
                t2 = S.comp[S.L[p + dir_off(4u + (i & 3u))] & 0x7FFFu];
            }
            if (t == b) t = t2;
            if (!RK_CHECK(t < nb, CK_BASIN)) continue;
            // both ends chose this edge: the lower number stays
            if (b < t && *(volatile uint32_t *)&S.best[t] == key && (S.sv[t] << 24 | K_SOURCE) < key) continue;
            S.up[b] = (uint16_t)t;
            S.capw[b] = (uint8_t)(key >> 24);
        }
        __syncthreads();
        // the live roots' new roots (the list and `ob` name no others), and what they bring along
#pragma unroll 1
        for (unsigned k = tid; k < nlive; k += NT) {
            const unsigned b = rounds ? now[k] : k + 1;
            unsigned t = b;
#pragma unroll 1
            for (unsigned u; (u = S.up[t]) != t;) t = u;
            if (t != b) {   // merged this round
                S.comp[b] = (uint16_t)t;
                atomicMax(&S.sv[t], S.sv[b]);
            } else if (S.best[b] < FINAL) {
                S.best[b] = 0u;
                const unsigned at = atomicAdd(&S.nlive[rounds & 1], 1u);
                if (RK_CHECK(at < (unsigned)Smem<CONN>::NB / (rounds & 1 ? 4 : 2), CK_LIVE)) next[at] = (uint16_t)b;
            }
        }
        __syncthreads();
        nlive = S.nlive[rounds & 1];
        if (nlive == 0) break;
    }

    // Per basin its cap (or final value) and node, cap << 8 | node slot, in comp.
    const unsigned nt = S.nt;
#pragma unroll 1
    for (unsigned b = tid; b < nb; b += NT) {
        unsigned v = 255u, root = b;
#pragma unroll 1
        for (unsigned t; (t = S.up[root]) != root; root = t) v = min(v, (unsigned)S.capw[root]);
        const bool node = S.best[root] == NODE;
        if (!node) v = min(v, (unsigned)S.capw[root]);
        S.comp[b] = (uint16_t)(v << 8 | (node ? S.capw[root] : RES));
        if (node && b == root) S.link[S.capw[b]] = S.sv[b] << 8 | RES;
    }
    __syncthreads();
    if (nt) {
        // Node links inside the block: to the source, then to each other. (An
        // edge left between two regions is no heavier than the caps inside them.)
        auto ends = [&](unsigned a, unsigned b, unsigned w) -> uint32_t {
            const unsigned fa = S.comp[a], fb = S.comp[b], na = fa & 255u, nb2 = fb & 255u;
            w = min(w, min(fa >> 8, fb >> 8));
            if (na == nb2 || w == 0) return 0u;
            if (na != RES && nb2 != RES) return na << 16 | nb2 << 8 | w;   // between two nodes
            if (RK_CHECK((na == RES ? nb2 : na) < nt, CK_SLOT)) atomicMax(&S.link[na == RES ? nb2 : na], w << 8 | RES);
            return 0u;
        };
        // (best and sv, next to each other, are no longer needed: room for every pass)
        uint32_t *const joins = S.best;
        static_assert(2 * Smem<CONN>::NB >= TAB && offsetof(Smem<CONN>, sv) == offsetof(Smem<CONN>, best) + sizeof(S.best), "joins");
        if (listed) {
#pragma unroll 1
            for (unsigned k = lane; k < mine; k += 32) {
                const uint32_t e = S.tab[seg0 + k], z = ends(e >> 20, (e >> 8) & 0xFFFu, e & 255u);
                if (!z) continue;
                const unsigned at = atomicAdd(&S.nj, 1u);   // gathered, so that whole warps join
                if (RK_CHECK(at < (unsigned)TAB, CK_PASS)) joins[at] = z;
            }
        } else {
            each_pair(S, [&](unsigned a, unsigned b, unsigned w, unsigned) { ends(a, b, w); });
        }
        __syncthreads();
        SharedLinks F{S.link, blk * MAX_TERM};
        bool ok = true;
        if (listed) {
            const unsigned nj = S.nj;
#pragma unroll 1
            for (unsigned i = tid; i < nj; i += NT) {
                const uint32_t e = joins[i];
                ok &= join(F, e >> 16, (e >> 8) & 255u, e & 255u);
            }
        } else {
            // (the sources' part was done above; links may now point to nodes)
            each_pair(S, [&](unsigned a, unsigned b, unsigned w, unsigned) {
                const unsigned fa = S.comp[a], fb = S.comp[b], na = fa & 255u, nb2 = fb & 255u;
                w = min(w, min(fa >> 8, fb >> 8));
                if (na != nb2 && na != RES && nb2 != RES && w) ok &= join(F, na, nb2, w);
            });
        }
        if (!ok) atomicCAS(&P.ctl->abort, 0, (int)rk::AB_MERGE);
        __syncthreads();
#pragma unroll 1
        for (unsigned k = tid; k < nt; k += NT) {
            const uint32_t l = S.link[k];
            const unsigned par = l & 255u;
            P.link[(size_t)blk * MAX_TERM + k] =
                (unsigned long long)(l >> 8) << 32 | (par == RES ? SRC : blk * MAX_TERM + par);
        }
    }
    if (tid == 0) P.block[blk] = Block{S.rec.tile, S.rec.local, S.rec.nbx, S.rec.nterm | nt};

    if (tid == 0) S.tick[4] = now_ns();
    // Results: the pixels themselves when everything is final, else (cap, node)
    const Tile &E = tile_of(P, S.tile);   // (read again: not kept in registers through the rounds)
    {
        const int cell = (r + 1) * ST + X0 + 16 * c;
        const uint2 i0 = *(const uint2 *)&bi[(r + 1) * IST + 2 + 4 * c], i1 = *(const uint2 *)&bi[(r + 1) * IST + 4 + 4 * c];
        const uint32_t iw[4] = {i0.x, i0.y, i1.x, i1.y};
        uint32_t o[8];   // 16 x (value << 8 | node slot)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint4 q = *(const uint4 *)&S.L[cell + 8 * h];
            const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {   // pixels 8h + 2j, 8h + 2j + 1
                const uint32_t i2 = iw[2 * h + (j >> 1)] >> (16 * (j & 1));
                o[4 * h + j] = RES | RES << 16;
                if (!RK_CHECK((w[j] & 0x7FFFu) < nb && (w[j] >> 16 & 0x7FFFu) < nb, CK_BASIN)) continue;
                const uint32_t e0 = S.comp[w[j] & 0x7FFFu], e1 = S.comp[(w[j] >> 16) & 0x7FFFu];
                o[4 * h + j] = (min(e0 >> 8, i2 & 255u) << 8 | (e0 & 255u)) |
                               (min(e1 >> 8, (i2 >> 8) & 255u) << 8 | (e1 & 255u)) << 16;
            }
        }
        if (nt == 0) {
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) w[j] = __byte_perm(o[2 * j], o[2 * j + 1], 0x7531) ^ (E.dual ? FULL : 0u);
            if (y < E.H) store16(E.J + (size_t)y * E.pitch + x, E.W - x, make_uint4(w[0], w[1], w[2], w[3]),
                                 (E.pitch % 16) == 0 && ((uintptr_t)E.J % 16) == 0);
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
        S.tick[5] = now_ns();
        rk::Work &wk = P.work[E.index];
        atomicAdd(&wk.visits, 1ull);
        atomicAdd(&wk.seeds, (unsigned long long)(nb - 1));
        atomicAdd(&wk.pops, (unsigned long long)ne);
        atomicAdd(&wk.levels, (unsigned long long)rounds + 1);
        atomicAdd(&wk.busy_ns, S.tick[5] - S.tick[0]);
#pragma unroll
        for (int k = 0; k < 5; ++k) atomicAdd(&wk.phase_ns[k], S.tick[k + 1] - S.tick[k]);
    }
}

// Joins across block borders: a CTA of 128 threads handles the edges from its
// block's right column (warps 0, 1) and bottom row (warps 2, 3) to the blocks
// E, NE, SE and S of it (the edges of its corners to NW and SW are the SE and NE
// edges of the blocks there). Bound by the latency of dependent loads (walks are 1
// to 6 links long on average, L2 accesses each), so everything before the walks
// takes two, and a lane whose neighbour holds the same two nodes with a heavier
// edge leaves it to that lane.
// 20 us on a 4096^2 h-dome tile, 27 us seeded from the border.
template <int CONN>
__global__ void __launch_bounds__(128) rim_kernel(const __grid_constant__ Params P)
{
    const unsigned blk = blockIdx.x;
    const bool right = threadIdx.x < 64;
    const int k = threadIdx.x & 63, lane = threadIdx.x & 31;
    allow_next();
    wait_previous();
    const Block B = P.block[blk];
    const unsigned pv = P.rim[(size_t)blk * 4 * BS + (right ? 3 * BS : BS) + k];
    if (!(B.nterm & (right ? B_RIGHT : B_DOWN))) return;   // warp-uniform
    const bool failed = P.tile_err[tile_of(P, B.tile).index] != 0;
    // opposite pixels k, k - 1, k + 1: their line in the block across, or a corner of the next one
    constexpr int ND = CONN == 8 ? 3 : 1;
    unsigned qn[ND], w[ND];
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        const int q = k + (d == 0 ? 0 : 2 * d - 3);
        unsigned nb = right ? blk + 1 : blk + B.nbx;
        int at = right ? 2 * BS + q : q;                  // left column / top row
        bool there = true;
        if (q < 0) {                                      // NE: its bottom row, x = 0
            there = right && (B.nterm & B_UP);
            nb = blk + 1 - B.nbx;
            at = BS;
        } else if (q >= BS) {                             // SE: its top row, x = 0
            there = right && (B.nterm & B_DOWN);
            nb = blk + 1 + B.nbx;
            at = 0;
        }
        there = there && RK_CHECK(nb < P.nblocks, CK_NODE);
        const unsigned qv = there ? P.rim[(size_t)nb * 4 * BS + at] : RES;
        qn[d] = (qv & 255u) == RES ? SRC : nb * MAX_TERM + (qv & 255u);
        w[d] = min(pv >> 8, qv >> 8);
    }
    if (failed) return;
    const unsigned pn = (pv & 255u) == RES ? SRC : blk * MAX_TERM + (pv & 255u);
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        if (pn == qn[d]) w[d] = 0;
#pragma unroll
        for (int e = 0; e < d; ++e)
            if (qn[e] == qn[d]) {
                w[e] = max(w[e], w[d]);
                w[d] = 0;
            }
    }
    GlobalLinks F{P.link, P.nblocks * MAX_TERM};
    bool ok = true;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        const unsigned pl = __shfl_up_sync(FULL, pn, 1), ql = __shfl_up_sync(FULL, qn[d], 1), wl = __shfl_up_sync(FULL, w[d], 1);
        const unsigned pr = __shfl_down_sync(FULL, pn, 1), qr = __shfl_down_sync(FULL, qn[d], 1),
                       wr = __shfl_down_sync(FULL, w[d], 1);
        if (lane > 0 && pl == pn && ql == qn[d] && wl >= w[d]) w[d] = 0;
        if (lane < 31 && pr == pn && qr == qn[d] && wr > w[d]) w[d] = 0;
    }
#pragma unroll 1
    for (int d = 0; d < ND; ++d) {
        const unsigned n = d == 0 ? qn[0] : (d == 1 ? qn[ND > 1 ? 1 : 0] : qn[ND > 2 ? 2 : 0]);
        const unsigned v = d == 0 ? w[0] : (d == 1 ? w[ND > 1 ? 1 : 0] : w[ND > 2 ? 2 : 0]);
        if (v) ok &= join(F, pn, n, v);
    }
    if (!ok) atomicCAS(&P.ctl->abort, 0, (int)rk::AB_MERGE);
}

// R of the block's nodes (the lightest link of their path to the source), then
// of its pixels.
__global__ void __launch_bounds__(NT) value_kernel(const __grid_constant__ Params P)
{
    __shared__ uint8_t R[256];
    const unsigned blk = blockIdx.x;
    const int r = threadIdx.x >> 2, c = threadIdx.x & 3;
    wait_previous();
    const Block B = P.block[blk];
    const unsigned nt = B.nterm & 255u;
    if (nt == 0) return;
    const uint4 *src = (const uint4 *)(P.px + (size_t)blk * BPX + r * BS + 16 * c);
    const uint4 q0 = src[0], q1 = src[1];
    const Tile D = tile_of(P, B.tile);
    R[threadIdx.x] = 255;
    if (threadIdx.x < nt) {
        unsigned n = blk * MAX_TERM + threadIdx.x, v = 255;
        int it = 0;
        for (; it < MAX_STEPS && RK_CHECK(n < P.nblocks * MAX_TERM, CK_NODE); ++it) {
            const unsigned long long l = __ldcg(&P.link[n]);
            v = min(v, (unsigned)(l >> 32));
            n = (unsigned)l;
            if (n == SRC) break;
        }
        if (it == MAX_STEPS) atomicCAS(&P.ctl->abort, 0, (int)rk::AB_MERGE);
        R[threadIdx.x] = (uint8_t)v;
    }
    __syncthreads();
    if (P.tile_err[D.index]) return;
    const int by = (int)(B.local / (unsigned)B.nbx), bx = (int)(B.local - (unsigned)by * B.nbx);
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
    store16(D.J + (size_t)y * D.pitch + x, D.W - x, make_uint4(w[0], w[1], w[2], w[3]), vec);
}

}  // namespace rf

RK_CHECK_READER(rf_read_checks)

extern "C" cudaError_t rf_configure()
{
    cudaError_t e = cudaFuncSetAttribute(rf::block_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(rf::Smem<8>));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(rf::block_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(rf::Smem<4>));
    return e;
}

// Launches kernel f behind the one before it on the stream, as its dependent.
template <class F>
static cudaError_t launch_after(F f, unsigned grid, int threads, const rf::Params *P, cudaStream_t st)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, f, *P);
}

extern "C" cudaError_t rf_launch(int conn, const rf::Params *P, cudaStream_t st)
{
    if (conn == 8) rf::block_kernel<8><<<P->nblocks, rf::NT, sizeof(rf::Smem<8>), st>>>(*P);
    else rf::block_kernel<4><<<P->nblocks, rf::NT, sizeof(rf::Smem<4>), st>>>(*P);
    cudaError_t e = cudaGetLastError();
    if (P->flat || e != cudaSuccess) return e;
    e = conn == 8 ? launch_after(rf::rim_kernel<8>, P->nblocks, 128, P, st) : launch_after(rf::rim_kernel<4>, P->nblocks, 128, P, st);
    if (e == cudaSuccess) e = launch_after(rf::value_kernel, P->nblocks, rf::NT, P, st);
    return e;
}
