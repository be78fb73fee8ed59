// Swendsen-Wang cluster updates of the Ising model on byte storage
// (Weigel & Yavors'kii 2011, Section 3: activate bonds between like spins with
// p = 1 - exp(-2 beta J), build the clusters joined by active bonds, flip each
// cluster with probability 1/2; cluster identification in tiles first, then
// amalgamation of the tiles through a union-and-find structure).
//
// One update is five kernels:
//   sw_local2, sw_local3
//               one CTA per tile (64 x 32 sites in 2D, 64 x 16 x 8 in 3D):
//               loads the tile's spins and a one-site halo on its +x/+y/+z
//               faces into shared memory (two words per row, by ballot, one lane
//               per site pair), draws the bond uniforms, joins each row's x-runs of
//               active bonds through warp ballots, then joins the runs along
//               y and z by a lock-free union-find in shared memory (the
//               larger root linked below the smaller by an atomic minimum),
//               which names every tile cluster by its smallest site (a y/z
//               bond is skipped when the bond beside it already joins the
//               same two runs), writes every site's label (the natural index
//               of its tile root, the smallest site of its tile cluster),
//               one bit per active bond that leaves the tile, and appends
//               its tile roots to a list;
//   sw_merge    one thread per tile-face bond: unites the two labels of each
//               active face bond in global memory (larger root below smaller);
//               afterwards the root of every cluster is its smallest site;
//   sw_resolve  one thread per listed tile root: follows the parents to the
//               cluster root g and rewrites the tile root's word as g with
//               g's flip bit (drawn from g's Philox output);
//   sw_flip     every site reads its tile root's word (its own word if it is
//               one) for the flip bit and flips;
//   sw_measure  E and M of the new configuration, closing the sweep.
// Label words: bits 0-29 the parent (a site index, N <= 2^30), bit 31 marks
// a tile root; after sw_resolve bit 30 of a tile root's word is its
// cluster's flip bit.  Every parent is a smaller or equal index and, beyond
// a site's first step, a tile root.
// Random numbers: the forward bond (i, i + e_mu) draws output 2 (i & 1) + mu
// of Philox(i >> 1, t, replica, 5 << 1) in 2D, output mu of
// Philox(i, t, replica, 5 << 1) in 3D; the cluster rooted at r flips iff the
// top bit of output 0 of Philox(r, t, replica, 6 << 1) is set.  Because the
// root is the smallest site whatever order the unions run in, the result does
// not depend on scheduling.
#include <cuda/atomic>

#include "internal.h"

namespace spinmc {
namespace {

constexpr uint32_t kSwBond = 5, kSwFlip = 6;
constexpr uint32_t kMask = 0x3FFFFFFFu;     // parent index
constexpr uint32_t kTileRoot = 0x80000000u;  // the site is a tile root
constexpr uint32_t kFlipBit = 0x40000000u;   // the cluster rooted here flips
constexpr int kSwThreads = 512;    // 3D tiles
constexpr int kSwThreads2 = 256;   // 2D tiles

template <int D>
struct SwTile;
template <>
struct SwTile<2> {
    static constexpr int TX = 64, TY = 32, TZ = 1;
};
template <>
struct SwTile<3> {
    static constexpr int TX = 64, TY = 16, TZ = 8;
};

template <int D>
struct SwFace {
    static constexpr int TX = SwTile<D>::TX, TY = SwTile<D>::TY, TZ = SwTile<D>::TZ;
    // face bits: +x face (TY x TZ), +y face (TX x TZ), +z face (TX x TY, 3D)
    static constexpr int BITS = TY * TZ + TX * TZ + (D == 3 ? TX * TY : 0);
    static constexpr int WORDS = BITS / 32;
};

struct SwArgs {
    int8_t* s[2];     // colour arrays (0 = up, 1 = down)
    uint32_t* lab;    // N labels, natural order
    uint32_t* face;   // WORDS per tile
    uint32_t* roots;  // the tile roots of an update (at most N), in no fixed order
    unsigned* nroots; // their number
    int L;
    int ntx, nty, ntz;
    FastDiv ntxd, ntyd;
    long long N, ntiles;
    uint32_t thr;     // a satisfied bond is active iff u <= thr
    int never;        // no bond can be active (beta = 0)
    int anti;         // J < 0: unlike spins satisfy a bond
    uint32_t replica;
    RoundKeys rk;
    Ctrl* ctrl;
};

int grid_for(long long work, int block)
{
    long long g = (work + block - 1) / block;
    if (g < 1) g = 1;
    if (g > kMaxBlocks) g = kMaxBlocks;
    return (int)g;
}

using gref = cuda::atomic_ref<uint32_t, cuda::thread_scope_device>;

__device__ __forceinline__ uint32_t gload(uint32_t* p)
{
    return gref(*p).load(cuda::memory_order_relaxed);
}

__device__ __forceinline__ void gstore(uint32_t* p, uint32_t v)
{
    gref(*p).store(v, cuda::memory_order_relaxed);
}

// global find with path halving (the same argument as in shared memory); a
// halving store keeps the entry's tile-root bit
__device__ __forceinline__ uint32_t gfind(uint32_t* lab, uint32_t x)
{
    uint32_t w = gload(lab + x);
    uint32_t p = w & kMask;
    while (p != x) {
        const uint32_t g = gload(lab + p) & kMask;
        if (g == p) return p;
        gstore(lab + x, g | (w & kTileRoot));
        x = g;
        w = gload(lab + x);
        p = w & kMask;
    }
    return x;
}

// roots are tile roots, so a root's word is r | kTileRoot
__device__ __forceinline__ void gunion(uint32_t* lab, uint32_t a, uint32_t b)
{
    a = gfind(lab, a);
    b = gfind(lab, b);
    while (a != b) {
        if (a < b) {
            const uint32_t t = a;
            a = b;
            b = t;
        }
        uint32_t expect = a | kTileRoot;
        if (gref(lab[a]).compare_exchange_strong(expect, b | kTileRoot,
                                                 cuda::memory_order_relaxed))
            return;
        a = gfind(lab, expect & kMask);
        b = gfind(lab, b);
    }
}


// origin and extents of tile (bx, by, bz)
template <int D>
__device__ __forceinline__ void tile_origin(const SwArgs& a, int bx, int by, int bz, int& X0, int& Y0,
                                            int& Z0, int& nx, int& ny, int& nz)
{
    constexpr int TX = SwTile<D>::TX, TY = SwTile<D>::TY, TZ = SwTile<D>::TZ;
    X0 = bx * TX;
    Y0 = by * TY;
    Z0 = bz * TZ;
    nx = min(TX, a.L - X0);
    ny = min(TY, a.L - Y0);
    nz = D == 3 ? min(TZ, a.L - Z0) : 1;
}

// root of x in the shared parent array, halving the path on the way (a
// halving store only ever replaces a non-root's parent by an ancestor)
__device__ __forceinline__ uint32_t sfind(volatile uint32_t* par, uint32_t x)
{
    uint32_t p = par[x];
    while (p != x) {
        const uint32_t g = par[p];
        if (g == p) return p;
        par[x] = g;
        x = g;
        p = par[x];
    }
    return x;
}

// 2D tiles of 64 x 32 sites.  A row of the tile is two words, the even and the
// odd sites' spins by ballot, and its four bond uniforms per site pair become
// four words of "drawn" bits by ballot, so bond activation, run heads, the choice
// of the bonds to unite and the tile's face are a few word operations per row for
// the whole warp.  (One lane deciding its own two sites' bonds byte by byte took
// 340 instructions per warp for its two rows and 46 of 252 us at L = 4096 at the
// critical point.)  Latency and issue bound: 256 threads and 8 blocks per
// multiprocessor (32 registers) took 178 us there, 512 threads 221 (3 blocks) and
// 193 (4 blocks), 128 threads 200, 1024 threads 245.
__global__ void __launch_bounds__(kSwThreads2, 8) sw_local2(const SwArgs a)
{
    constexpr int TX = SwTile<2>::TX, TY = SwTile<2>::TY;
    constexpr int NW = kSwThreads2 / 32, RPW = TY / NW;  // warps, rows per warp
    constexpr uint32_t kAll = 0xFFFFFFFFu;
    static_assert(TX == 64 && TY == 32, "words of a tile");
    __shared__ __align__(8) uint32_t par[TX * TY];
    __shared__ uint32_t rowE[TY + 1], rowO[TY + 1];  // spins, with the row after the tile
    __shared__ uint32_t bx0[TY], bx1[TY];            // active x bonds of even and odd sites
    __shared__ uint32_t fx;                          // bonds over the +x face
    __shared__ uint16_t list[NW][RPW * TX];
    __shared__ unsigned blk_count, blk_base;

    int X0, Y0, Z0, nx, ny, nz;
    // (one block per tile on a grid of the tiles' shape: recovering the tile from a
    // linear index took three 64-bit divisions, some 250 instructions a thread)
    tile_origin<2>(a, blockIdx.x, blockIdx.y, 0, X0, Y0, Z0, nx, ny, nz);
    const size_t tile = blockIdx.x + (size_t)gridDim.x * blockIdx.y;
    const uint32_t L = (uint32_t)a.L;
    const uint32_t t = (uint32_t)a.ctrl->t;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lx0 = 2 * lane, last = (nx >> 1) - 1;  // the lane's pair; lane of the last pair
    const uint32_t valid = kAll >> (31 - last), below = (1u << lane) - 1u;
    const bool ex = lane <= last;
    if (threadIdx.x == 0) {
        fx = 0u;
        blk_count = 0;
    }

    // spins of row ly of the tile (up to ny, the row after it)
    auto load_row = [&](int ly) {
        const uint32_t y = (uint32_t)(Y0 + ly) == L ? 0u : (uint32_t)(Y0 + ly);
        const int ce = (int)(y & 1u);  // colour of the even-x sites
        const uint32_t j = (L * y + (uint32_t)(X0 + lx0)) >> 1;
        const int8_t ve = ex ? a.s[ce][j] : (int8_t)0, vo = ex ? a.s[ce ^ 1][j] : (int8_t)0;
        const uint32_t E = __ballot_sync(kAll, ve != 0), O = __ballot_sync(kAll, vo != 0);
        if (lane == 0) {
            rowE[ly] = E;
            rowO[ly] = O;
        }
    };
    uint32_t hx = 0u;  // bit k: the spin after the last of the warp's row k
#pragma unroll
    for (int k = 0; k < RPW; ++k) {
        const int ly = RPW * warp + k;
        if (ly >= ny) continue;  // uniform across the warp
        load_row(ly);
        const uint32_t y = (uint32_t)(Y0 + ly), x = (uint32_t)(X0 + nx) == L ? 0u : (uint32_t)(X0 + nx);
        hx |= (uint32_t)a.s[(x + y) & 1u][(L * y + x) >> 1] << k;
    }
    if (warp == NW - 1) load_row(ny);
    // drawn bits of the x and y bonds of the even and odd sites (the draws have no
    // branch between them; rows outside a ragged tile draw bits nobody reads)
    uint32_t ax0[RPW], ax1[RPW], ay0[RPW], ay1[RPW];
    {
        const PhiloxGroups pg = philox_groups(t, a.replica, kSwBond << 1, a.rk);
        uint4 rnd[RPW];
#pragma unroll
        for (int k = 0; k < RPW; ++k)
            rnd[k] = philox_at(pg, ((uint32_t)(X0 + lx0) + L * (uint32_t)(Y0 + RPW * warp + k)) >> 1,
                               a.rk);
        const uint32_t may = a.never ? 0u : valid;
#pragma unroll
        for (int k = 0; k < RPW; ++k) {
            ax0[k] = __ballot_sync(kAll, rnd[k].x <= a.thr) & may;
            ay0[k] = __ballot_sync(kAll, rnd[k].y <= a.thr) & may;
            ax1[k] = __ballot_sync(kAll, rnd[k].z <= a.thr) & may;
            ay1[k] = __ballot_sync(kAll, rnd[k].w <= a.thr) & may;
        }
    }
    __syncthreads();

    // Active bonds, and every site's parent: the first site of its x-run.
    const uint32_t flipw = a.anti ? 0u : kAll;  // like spins satisfy a bond, or unlike ones
#pragma unroll
    for (int k = 0; k < RPW; ++k) {
        const int ly = RPW * warp + k;
        if (ly >= ny) {
            ay0[k] = ay1[k] = ax0[k] = ax1[k] = 0u;
            continue;
        }
        const uint32_t E = rowE[ly], O = rowO[ly];
        ax0[k] &= E ^ O ^ flipw;
        ax1[k] &= O ^ ((E >> 1) | ((hx >> k & 1u) << last)) ^ flipw;
        ay0[k] &= E ^ rowE[ly + 1] ^ flipw;
        ay1[k] &= O ^ rowO[ly + 1] ^ flipw;
        if (lane == 0 && (ax1[k] >> last & 1u)) atomicOr(&fx, 1u << ly);
        ax1[k] &= ~(1u << last);
        if (ly + 1 == ny) {  // the +y face
            uint32_t* f = a.face + tile * SwFace<2>::WORDS;
            if (lane < 2) f[1 + lane] = lane ? ay1[k] : ay0[k];
            ay0[k] = ay1[k] = 0u;
        }
        if (lane == 0) {
            bx0[ly] = ax0[k];
            bx1[ly] = ax1[k];
        }
        // run starts: the even site unless the bond from the previous lane's odd
        // site is active, the odd site unless the pair's bond is
        const uint32_t R0 = ~(ax1[k] << 1), R1 = ~ax0[k];
        int rs0 = 2 * (31 - __clz(R0 & ((2u << lane) - 1u)));
        const uint32_t m1 = R1 & below;
        if (m1) rs0 = max(rs0, 2 * (31 - __clz(m1)) + 1);
        const int rs1 = (ax0[k] >> lane & 1u) ? rs0 : lx0 + 1;
        *reinterpret_cast<uint2*>(&par[TX * ly + lx0]) =
            make_uint2((uint32_t)(TX * ly + rs0), (uint32_t)(TX * ly + rs1));
    }
    __syncthreads();

    // place the sites of two masks (even, odd) of row ly in the warp's list
    auto put = [&](uint32_t m0, uint32_t m1, int ly, unsigned& n) {
        const unsigned n0 = __popc(m0);
        if (m0 >> lane & 1u) list[warp][n + __popc(m0 & below)] = (uint16_t)(TX * ly + lx0);
        if (m1 >> lane & 1u) list[warp][n + n0 + __popc(m1 & below)] = (uint16_t)(TX * ly + lx0 + 1);
        n += n0 + __popc(m1);
    };
    // The runs are joined along y.  A bond is left out when the two runs are
    // joined by a bond further left already: c0, c1 mark the even and odd sites
    // whose left neighbour is joined to its lower one, in both rows to the site.
    // First come the bonds within the warp's rows (within pairs of rows, then
    // between the pairs), then those to the next warp's.
    unsigned n = 0, inner = 0;
#pragma unroll
    for (int kk = 0; kk < RPW; ++kk) {
        const int k = kk == 1 ? 2 : kk == 2 ? 1 : kk;
        const int ly = RPW * warp + k;
        if (k == RPW - 1) inner = n;
        if (ly + 1 >= ny) continue;
        const uint32_t r0 = ax0[k] & bx0[ly + 1], r1 = (ax1[k] & bx1[ly + 1]) << 1;
        uint32_t c0 = 0u, c1 = 0u;
#pragma unroll
        for (int it = 0; it < 3; ++it) {
            c1 = (ay0[k] | c0) & r0;
            c0 = (ay1[k] | c1) << 1 & r1;
        }
        put(ay0[k] & ~c0, ay1[k] & ~c1, ly, n);
    }
    __syncwarp();
    // One union per remaining bond, lock-free, the bonds dealt out evenly over the
    // warp: find both roots (path halving) and link the larger below the smaller by
    // an atomic minimum; if another link got there first, what it linked to is
    // still to be joined to the smaller root.  Parents only ever point to smaller
    // indices, so the root of every tile cluster ends as its smallest site whatever
    // order the unions run in; but the order decides how long the paths grow.  A warp
    // has four rows that follow each other and joins them before any warp joins its
    // rows to the next one's: the whole update took 995 us at L = 8192 with every
    // eighth row to a warp, 886 with four rows on end, 870 with the barrier.
    // (Measured for the whole kernel up to here at L = 4096, critical point, every
    // eighth row: compare-and-swap with both finds repeated 171 us, atomic minimum
    // 163, Rem's interleaved splicing 161 but dearer jumps after it; finds without
    // halving 1.4 times the whole kernel.)
    volatile uint32_t* vp = par;
    auto unite = [&](unsigned q, unsigned end) {
        for (; q < end; q += 32) {
            const uint32_t u = list[warp][q];
            uint32_t ra = sfind(vp, u), rb = sfind(vp, u + (uint32_t)TX);
            while (ra != rb) {
                const uint32_t hi = max(ra, rb), lo = min(ra, rb);
                const uint32_t old = atomicMin(par + hi, lo);
                if (old == hi) break;
                ra = sfind(vp, old);
                rb = lo;
            }
        }
    };
    unite(lane, inner);
    __syncthreads();
    unite(inner + lane, n);
    // the run heads, listed in the same place, jump to their roots; every other
    // site's label is read through its head
    __syncwarp();
    unsigned nh = 0;
#pragma unroll
    for (int k = 0; k < RPW; ++k) {
        const int ly = RPW * warp + k;
        if (ly < ny) put(~(ax1[k] << 1) & valid, ~ax0[k] & valid, ly, nh);
    }
    __syncthreads();
    for (unsigned q = lane; q < nh; q += 32) {
        const uint32_t l = list[warp][q];
        uint32_t p = vp[l];
        while (true) {
            const uint32_t g = vp[p];
            if (g == p) break;
            p = g;
        }
        vp[l] = p;
    }
    __syncthreads();

    // labels: the natural index of each site's tile root; tile roots are marked
    // and appended to the update's list (one global atomic per block)
    const uint32_t i00 = (uint32_t)X0 + L * (uint32_t)Y0;
    uint32_t m0[RPW], m1[RPW];  // tile roots among the even and odd sites
    unsigned cnt = 0;
#pragma unroll
    for (int k = 0; k < RPW; ++k) {
        const int ly = RPW * warp + k;
        m0[k] = m1[k] = 0u;
        if (ly >= ny) continue;
        const uint32_t l = (uint32_t)(TX * ly + lx0);
        const uint2 h = ex ? *reinterpret_cast<const uint2*>(&par[l]) : make_uint2(l, l);
        const uint32_t ra = par[h.x], rb = par[h.y];
        const bool root0 = ex && ra == l, root1 = ex && rb == l + 1;
        m0[k] = __ballot_sync(kAll, root0);
        m1[k] = __ballot_sync(kAll, root1);
        cnt += __popc(m0[k]) + __popc(m1[k]);
        if (ex)
            *reinterpret_cast<uint2*>(a.lab + i00 + L * (uint32_t)ly + lx0) =
                make_uint2((i00 + (ra & 63u) + L * (ra >> 6)) | (root0 ? kTileRoot : 0u),
                           (i00 + (rb & 63u) + L * (rb >> 6)) | (root1 ? kTileRoot : 0u));
    }
    unsigned pos = 0;
    if (lane == 0) pos = atomicAdd(&blk_count, cnt);
    __syncthreads();
    if (threadIdx.x == 0) {
        blk_base = atomicAdd(a.nroots, blk_count);
        a.face[tile * SwFace<2>::WORDS] = fx;
    }
    __syncthreads();
    pos = blk_base + __shfl_sync(kAll, pos, 0);
#pragma unroll
    for (int k = 0; k < RPW; ++k) {
        const uint32_t i = i00 + L * (uint32_t)(RPW * warp + k) + lx0;
        if (m0[k] >> lane & 1u) a.roots[pos + __popc(m0[k] & below)] = i;
        pos += __popc(m0[k]);
        if (m1[k] >> lane & 1u) a.roots[pos + __popc(m1[k] & below)] = i + 1;
        pos += __popc(m1[k]);
    }
}

// 3D tiles of 64 x 16 x 8 sites, by words as in 2D: a warp has eight rows on end,
// half of a plane.  It joins them along y first; then the rows are joined to the next
// warp's and along z.  (A lane deciding its own sites' bonds from bytes and uniting
// them one after another, every sixteenth row to a warp: an update at L = 256 took 450
// us at the critical point, 497 at beta = 0.4 and 405 at 0.15, now 428, 466 and 406;
// L = 100 98 and 89.  Issue bound; 2 and 4 blocks a multiprocessor: 462 and 423 at L =
// 256, 87 and 90 at L = 100.)
__global__ void __launch_bounds__(kSwThreads, 3) sw_local3(const SwArgs a)
{
    constexpr int TX = SwTile<3>::TX, TY = SwTile<3>::TY, TZ = SwTile<3>::TZ;
    constexpr int HY = TY + 1, HZ = TZ + 1;  // rows with those after the tile
    constexpr int WORDS = SwFace<3>::WORDS;
    constexpr int NW = kSwThreads / 32, ROWS = TY * TZ, RPW = ROWS / NW;
    constexpr uint32_t kAll = 0xFFFFFFFFu;
    static_assert(TX == 64 && RPW == 8 && TY % RPW == 0, "rows of a warp");
    __shared__ __align__(8) uint32_t par[TX * ROWS];
    __shared__ uint32_t rowE[HZ * HY], rowO[HZ * HY];  // spins of even and odd sites
    __shared__ uint32_t bx[2][ROWS], by[2][ROWS], bz[2][ROWS];  // active bonds in the tile
    __shared__ uint32_t fm[WORDS];
    __shared__ uint16_t list[NW][5 * TX];
    __shared__ unsigned blk_count, blk_base;

    const size_t tile = blockIdx.x + gridDim.x * (blockIdx.y + (size_t)gridDim.y * blockIdx.z);
    int X0, Y0, Z0, nx, ny, nz;
    tile_origin<3>(a, blockIdx.x, blockIdx.y, blockIdx.z, X0, Y0, Z0, nx, ny, nz);
    const uint32_t L = (uint32_t)a.L;
    const uint32_t t = (uint32_t)a.ctrl->t;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lx0 = 2 * lane, last = (nx >> 1) - 1;  // the lane's pair; lane of the last pair
    const uint32_t valid = kAll >> (31 - last), below = (1u << lane) - 1u;
    const bool ex = lane <= last;
    const int row0 = RPW * warp, ly0 = row0 % TY, lz = row0 / TY;  // the warp's first row
    // the rows of the warp that lie in the tile
    const int rows = lz >= nz || ly0 >= ny ? 0 : min(RPW, ny - ly0);
    const uint32_t zb = L * (L * (uint32_t)(Z0 + lz) + (uint32_t)(Y0 + ly0));  // its row's first site

    for (int w = threadIdx.x; w < WORDS; w += kSwThreads) fm[w] = 0u;
    if (threadIdx.x == 0) blk_count = 0;
    // the tile's rows, the +y row and the +z plane (one warp per row)
    for (int r = warp; r < HY * HZ; r += NW) {
        const int hy = r % HY, hz = r / HY;
        if (hy > ny || hz > nz || (hy == ny && hz == nz)) continue;
        const uint32_t y = (uint32_t)(Y0 + hy) == L ? 0u : (uint32_t)(Y0 + hy);
        const uint32_t z = (uint32_t)(Z0 + hz) == L ? 0u : (uint32_t)(Z0 + hz);
        const int ce = (int)((y + z) & 1u);  // colour of the even-x sites
        const uint32_t j = (L * (y + L * z) + (uint32_t)(X0 + lx0)) >> 1;
        const int8_t ve = ex ? a.s[ce][j] : (int8_t)0, vo = ex ? a.s[ce ^ 1][j] : (int8_t)0;
        const uint32_t E = __ballot_sync(kAll, ve != 0), O = __ballot_sync(kAll, vo != 0);
        if (lane == 0) {
            rowE[r] = E;
            rowO[r] = O;
        }
    }
    uint32_t hx = 0u;  // bit k: the spin after the last of the warp's row k
    {
        const uint32_t x = (uint32_t)(X0 + nx) == L ? 0u : (uint32_t)(X0 + nx);
        for (int k = 0; k < rows; ++k)
            hx |= (uint32_t)a.s[(x + (uint32_t)(Y0 + ly0 + k + Z0 + lz)) & 1u]
                               [(zb + L * (uint32_t)k + x) >> 1] << k;
    }
    __syncthreads();

    // Active bonds, and every site's parent: the first site of its x-run.  Bonds that
    // leave the tile go to its face words (even sites' word, odd sites' word).
    {
        const PhiloxGroups pg = philox_groups(t, a.replica, kSwBond << 1, a.rk);
        const uint32_t may = a.never ? 0u : valid;
        const uint32_t flipw = a.anti ? 0u : kAll;  // like spins satisfy a bond, or unlike ones
        uint32_t fxw = 0u;
#pragma unroll 2
        for (int k = 0; k < rows; ++k) {
            const int row = row0 + k, ly = ly0 + k, r = lz * HY + ly;
            const uint32_t i0 = zb + L * (uint32_t)k + (uint32_t)(X0 + lx0);
            const uint4 u0 = philox_at(pg, i0, a.rk), u1 = philox_at(pg, i0 + 1u, a.rk);
            const uint32_t E = rowE[r], O = rowO[r];
            const uint32_t x0 = __ballot_sync(kAll, u0.x <= a.thr) & may & (E ^ O ^ flipw);
            uint32_t x1 = __ballot_sync(kAll, u1.x <= a.thr) & may &
                          (O ^ ((E >> 1) | ((hx >> k & 1u) << last)) ^ flipw);
            uint32_t y0 = __ballot_sync(kAll, u0.y <= a.thr) & may & (E ^ rowE[r + 1] ^ flipw);
            uint32_t y1 = __ballot_sync(kAll, u1.y <= a.thr) & may & (O ^ rowO[r + 1] ^ flipw);
            uint32_t z0 = __ballot_sync(kAll, u0.z <= a.thr) & may & (E ^ rowE[r + HY] ^ flipw);
            uint32_t z1 = __ballot_sync(kAll, u1.z <= a.thr) & may & (O ^ rowO[r + HY] ^ flipw);
            fxw |= (x1 >> last & 1u) << (row & 31);
            x1 &= ~(1u << last);
            if (ly + 1 == ny) {
                if (lane < 2) fm[ROWS / 32 + 2 * lz + lane] = lane ? y1 : y0;
                y0 = y1 = 0u;
            }
            if (lz + 1 == nz) {
                if (lane < 2) fm[(ROWS + TX * TZ) / 32 + 2 * ly + lane] = lane ? z1 : z0;
                z0 = z1 = 0u;
            }
            if (lane == 0) {
                bx[0][row] = x0;
                bx[1][row] = x1;
                by[0][row] = y0;
                by[1][row] = y1;
                bz[0][row] = z0;
                bz[1][row] = z1;
            }
            // run starts: the even site unless the bond from the previous lane's odd
            // site is active, the odd site unless the pair's bond is
            const uint32_t R0 = ~(x1 << 1), R1 = ~x0;
            int rs0 = 2 * (31 - __clz(R0 & ((2u << lane) - 1u)));
            const uint32_t m1 = R1 & below;
            if (m1) rs0 = max(rs0, 2 * (31 - __clz(m1)) + 1);
            const int rs1 = (x0 >> lane & 1u) ? rs0 : lx0 + 1;
            *reinterpret_cast<uint2*>(&par[TX * row + lx0]) =
                make_uint2((uint32_t)(TX * row + rs0), (uint32_t)(TX * row + rs1));
        }
        if (lane == 0 && fxw) atomicOr(&fm[row0 >> 5], fxw);
    }
    __syncthreads();

    // place the sites of two masks (even, odd) of a row in the warp's list
    auto put = [&](uint32_t m0, uint32_t m1, int row, unsigned& n) {
        const unsigned n0 = __popc(m0);
        if (m0 >> lane & 1u) list[warp][n + __popc(m0 & below)] = (uint16_t)(TX * row + lx0);
        if (m1 >> lane & 1u)
            list[warp][n + n0 + __popc(m1 & below)] = (uint16_t)(TX * row + lx0 + 1);
        n += n0 + __popc(m1);
    };
    // the bonds w between the warp's row k and the one `step` rows on, without those
    // whose two runs a bond further left has joined already (see sw_local2)
    auto put_bonds = [&](const uint32_t (&w)[2][ROWS], int k, int step, unsigned& n) {
        if (k >= rows) return;
        const int row = row0 + k, next = min(row + step, ROWS - 1);
        const uint32_t w0 = w[0][row], w1 = w[1][row];
        const uint32_t r0 = bx[0][row] & bx[0][next], r1 = (bx[1][row] & bx[1][next]) << 1;
        uint32_t c0 = 0u, c1 = 0u;
#pragma unroll
        for (int it = 0; it < 3; ++it) {
            c1 = (w0 | c0) & r0;
            c0 = (w1 | c1) << 1 & r1;
        }
        put(w0 & ~c0, w1 & ~c1, row, n);
    };
    // one union per listed bond, the first ny of them along y (see sw_local2)
    volatile uint32_t* vp = par;
    auto unite = [&](unsigned n, unsigned ny_) {
        __syncwarp();
        for (unsigned q = lane; q < n; q += 32) {
            const uint32_t u = list[warp][q];
            const uint32_t v = u + (uint32_t)(q < ny_ ? TX : TX * TY);
            uint32_t ra = sfind(vp, u), rb = sfind(vp, v);
            while (ra != rb) {
                const uint32_t hi = max(ra, rb), lo = min(ra, rb);
                const uint32_t old = atomicMin(par + hi, lo);
                if (old == hi) break;
                ra = sfind(vp, old);
                rb = lo;
            }
        }
        __syncwarp();
    };
    unsigned n = 0;
    for (int k = 0; k < RPW; k += 2) put_bonds(by, k, 1, n);
    unite(n, n);
    n = 0;
    for (int k = 1; k < RPW - 1; k += 2) put_bonds(by, k, 1, n);
    unite(n, n);
    __syncthreads();
    n = 0;
    put_bonds(by, RPW - 1, 1, n);
    const unsigned along_y = n;
    for (int k = 0; k < 4; ++k) put_bonds(bz, k, TY, n);
    unite(n, along_y);
    n = 0;
    for (int k = 4; k < RPW; ++k) put_bonds(bz, k, TY, n);
    unite(n, 0u);
    __syncthreads();
    // the run heads jump to their roots; every other site's label is read through
    // its head
    for (int k = 0; k < rows; k += 4) {
        n = 0;
        for (int q = k; q < k + 4 && q < rows; ++q)
            put(~(bx[1][row0 + q] << 1) & valid, ~bx[0][row0 + q] & valid, row0 + q, n);
        __syncwarp();
        for (unsigned q = lane; q < n; q += 32) {
            const uint32_t l = list[warp][q];
            uint32_t p = vp[l];
            while (true) {
                const uint32_t g = vp[p];
                if (g == p) break;
                p = g;
            }
            vp[l] = p;
        }
        __syncwarp();
    }
    __syncthreads();

    // labels: the natural index of each site's tile root; tile roots are marked
    // and appended to the update's list (one global atomic per block)
    const uint32_t i00 = (uint32_t)X0 + L * ((uint32_t)Y0 + L * (uint32_t)Z0);
    auto label = [&](uint32_t m) {
        return i00 + (m & 63u) + L * ((m >> 6 & 15u) + L * (m >> 10));
    };
    uint32_t mine = 0u;  // bits 2 k, 2 k + 1: the lane's sites of row k are tile roots
#pragma unroll 4
    for (int k = 0; k < rows; ++k) {
        if (!ex) continue;
        const uint32_t l = (uint32_t)(TX * (row0 + k) + lx0);
        const uint2 h = *reinterpret_cast<const uint2*>(&par[l]);
        const uint32_t ra = par[h.x], rb = par[h.y];
        const uint32_t root0 = ra == l, root1 = rb == l + 1;
        mine |= (root0 | root1 << 1) << (2 * k);
        *reinterpret_cast<uint2*>(a.lab + zb + L * (uint32_t)k + (uint32_t)(X0 + lx0)) =
            make_uint2(label(ra) | (root0 ? kTileRoot : 0u), label(rb) | (root1 ? kTileRoot : 0u));
    }
    for (int w = threadIdx.x; w < WORDS; w += kSwThreads) a.face[tile * WORDS + w] = fm[w];
    const unsigned cnt = __popc(mine);
    unsigned incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(kAll, incl, o);
        if (lane >= o) incl += v;
    }
    unsigned wbase = 0;
    if (lane == 31) wbase = atomicAdd(&blk_count, incl);
    wbase = __shfl_sync(kAll, wbase, 31);
    __syncthreads();
    if (threadIdx.x == 0) blk_base = atomicAdd(a.nroots, blk_count);
    __syncthreads();
    unsigned pos = blk_base + wbase + incl - cnt;
    for (uint32_t bits = mine; bits; bits &= bits - 1) {
        const int bit = __ffs(bits) - 1;
        a.roots[pos++] = zb + L * (uint32_t)(bit >> 1) + (uint32_t)(X0 + lx0 + (bit & 1));
    }
}

template <int D>
__global__ void __launch_bounds__(256) sw_merge(const SwArgs a)
{
    constexpr int TX = SwTile<D>::TX, TY = SwTile<D>::TY, TZ = SwTile<D>::TZ;
    constexpr int WORDS = SwFace<D>::WORDS;
    // (N <= 2^30 keeps the number of face bits below 2^31)
    const uint32_t total = (uint32_t)(a.ntiles * WORDS * 32);
    const int L = a.L;
    for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < total;
         q += gridDim.x * blockDim.x) {
        const uint32_t b = q / (WORDS * 32);
        const int bit = (int)(q % (WORDS * 32));
        const uint32_t word = __ldg(a.face + (size_t)b * WORDS + (bit >> 5));
        if (!((word >> (bit & 31)) & 1u)) continue;
        const uint32_t brow = a.ntxd.div(b);
        const uint32_t bz = D == 3 ? a.ntyd.div(brow) : 0u;
        int X0, Y0, Z0, nx, ny, nz;
        tile_origin<D>(a, (int)(b - brow * a.ntxd.d),
                       (int)(D == 3 ? brow - bz * a.ntyd.d : brow), (int)bz, X0, Y0, Z0, nx, ny, nz);
        int lx, ly, lz, mu;
        if (bit < TY * TZ) {
            mu = 0;
            lx = nx - 1;
            ly = bit % TY;
            lz = bit / TY;
        } else if (bit < TY * TZ + TX * TZ) {
            mu = 1;
            // (per row the even sites' word, then the odd sites')
            const int k = bit - TY * TZ;
            lx = 2 * (k & 31) + (k >> 5 & 1);
            ly = ny - 1;
            lz = k / TX;
        } else {
            mu = 2;
            const int k = bit - TY * TZ - TX * TZ;
            lx = 2 * (k & 31) + (k >> 5 & 1);
            ly = k / TX;
            lz = nz - 1;
        }
        const int x = X0 + lx, y = Y0 + ly, z = Z0 + lz;
        int xn = x, yn = y, zn = z;
        if (mu == 0) xn = x + 1 == L ? 0 : x + 1;
        if (mu == 1) yn = y + 1 == L ? 0 : y + 1;
        if (mu == 2) zn = z + 1 == L ? 0 : z + 1;
        const uint32_t i = (uint32_t)x + (uint32_t)L * ((uint32_t)y + (uint32_t)L * (uint32_t)z);
        const uint32_t j = (uint32_t)xn + (uint32_t)L * ((uint32_t)yn + (uint32_t)L * (uint32_t)zn);
        gunion(a.lab, i, j);
    }
}

// One thread per listed tile root: follow the parents to the cluster root g
// (the smallest site of the cluster) and rewrite the tile root's word as g
// with g's flip bit, the top bit of output 0 of Philox(g, t, replica, 6 << 1).
// Tile roots are each other's parents, so a chase may read a word another
// thread has just rewritten; the new word points at g itself, so the chase
// still ends at g.
__global__ void __launch_bounds__(256) sw_resolve(const SwArgs a)
{
    const uint32_t t = (uint32_t)a.ctrl->t;
    const unsigned n = *a.nroots;
    const unsigned stride = gridDim.x * blockDim.x;
    // two roots per pass with their chases interleaved, so each thread keeps
    // two dependent load chains in flight (a missing second root repeats the
    // first and stores nothing)
    for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += 2 * stride) {
        const bool two = q + stride < n;
        const uint32_t r0 = __ldcg(a.roots + q);
        const uint32_t r1 = two ? __ldcg(a.roots + q + stride) : r0;
        uint32_t p0 = gload(a.lab + r0) & kMask, p1 = gload(a.lab + r1) & kMask;
        while (true) {
            const uint32_t g0 = gload(a.lab + p0) & kMask;
            const uint32_t g1 = gload(a.lab + p1) & kMask;
            if (g0 == p0 && g1 == p1) break;
            p0 = g0;
            p1 = g1;
        }
        const uint4 rnd0 = philox4x32_10(make_uint4(p0, t, a.replica, kSwFlip << 1), a.rk);
        const uint4 rnd1 = philox4x32_10(make_uint4(p1, t, a.replica, kSwFlip << 1), a.rk);
        gstore(a.lab + r0, p0 | kTileRoot | ((rnd0.x >> 31) ? kFlipBit : 0u));
        if (two) gstore(a.lab + r1, p1 | kTileRoot | ((rnd1.x >> 31) ? kFlipBit : 0u));
    }
}

// flip bit of site i's cluster from its label word l: a tile root carries it,
// any other site's parent is its tile root
__device__ __forceinline__ uint32_t root_bit(const SwArgs& a, uint32_t i, uint32_t l)
{
    const uint32_t word = (l & kTileRoot) ? l : __ldg(a.lab + (l & kMask));
    return (word & kFlipBit) ? 1u : 0u;
}

// Every site flips iff its cluster's root drew the flip bit.  A thread takes
// four site pairs (x even, x + 1): eight labels and one 32-bit word of each
// colour array.
// Threads of a block share rows: tq threads per row (the whole block on a
// long row), so the row's coordinates and colour come from one division per
// row rather than per word.
struct RowSplit {
    int tq, rpb, rsub, q0;
    __device__ RowSplit(int Q)
    {
        tq = Q >= (int)blockDim.x ? (int)blockDim.x : Q;
        rpb = (int)blockDim.x / tq;
        rsub = (int)threadIdx.x / tq;
        q0 = (int)threadIdx.x - rsub * tq;
    }
};

__global__ void __launch_bounds__(256) sw_flip(const SwArgs a)
{
    const long long H = a.N >> 1;
    const int L = a.L, W = L >> 1;
    if ((W & 3) == 0) {
        // rows of W colour entries, 4 per word of each colour array; the
        // labels of the 8 sites of word q are the uint4 pair 2q, 2q + 1
        const int Q = W >> 2;
        const long long rows = H / W;
        const RowSplit rs(Q);
        if (rs.rsub >= rs.rpb) return;
        for (long long row = (long long)blockIdx.x * rs.rpb + rs.rsub; row < rows;
             row += (long long)gridDim.x * rs.rpb) {
            const bool c0 = ((row % L + row / L) & 1) != 0;  // colour of the even sites
            for (int qi = rs.q0; qi < Q; qi += rs.tq) {
                const long long q = row * Q + qi;
                const uint4 la = __ldg(reinterpret_cast<const uint4*>(a.lab) + 2 * q);
                const uint4 lb = __ldg(reinterpret_cast<const uint4*>(a.lab) + 2 * q + 1);
                const uint32_t lw[8] = {la.x, la.y, la.z, la.w, lb.x, lb.y, lb.z, lb.w};
                const uint32_t i0 = (uint32_t)(8 * q);
                uint32_t fl0 = 0u, fl1 = 0u;  // flips of colour 0 / colour 1 bytes
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t fe = root_bit(a, i0 + 2 * e, lw[2 * e]) << (8 * e);
                    const uint32_t fo = root_bit(a, i0 + 2 * e + 1, lw[2 * e + 1]) << (8 * e);
                    fl0 |= c0 ? fo : fe;
                    fl1 |= c0 ? fe : fo;
                }
                if (fl0) reinterpret_cast<uint32_t*>(a.s[0])[q] ^= fl0;
                if (fl1) reinterpret_cast<uint32_t*>(a.s[1])[q] ^= fl1;
            }
        }
        return;
    }
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < H;
         j += (long long)gridDim.x * blockDim.x) {
        const long long i0 = 2 * j;
        const long long row = i0 / L;
        const int c0 = (int)((row % L + row / L) & 1);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const uint32_t i = (uint32_t)(i0 + e);
            const int8_t f = (int8_t)root_bit(a, i, __ldg(a.lab + i));
            int8_t* sp = a.s[c0 ^ e] + j;
            *sp = (int8_t)(*sp ^ f);
        }
    }
}

// E and M after an update, streaming 32-bit words (four colour-1 sites) of
// every colour-1 row against the colour-0 rows around it; closes the sweep
// like every other measured pass (series entry, sweep counter + 1).  Needs
// L % 8 == 0.  Every bond touches exactly one colour-1 site, so the bond sum
// is sum over colour-1 sites of 2d - 2 (unlike neighbours).
template <int D>
__global__ void __launch_bounds__(256) sw_measure(const SwArgs a, Partial* partials, double J)
{
    __shared__ long long red[32];
    const int L = a.L, W = L / 2, Q = W / 4;
    const long long rows = (long long)L * (D == 3 ? L : 1);
    const uint32_t* own = reinterpret_cast<const uint32_t*>(a.s[1]);
    const uint32_t* oth = reinterpret_cast<const uint32_t*>(a.s[0]);
    const uint32_t ones = 0x01010101u;
    long long bond = 0, down = 0;
    // one site word: A own, cur the other colour's word at the same place,
    // S its x-shifted neighbour word, nv the y (and z) neighbour words
    auto word = [&](uint32_t A, uint32_t cur, uint32_t S, uint32_t nv) {
        const uint32_t nd = cur + S + nv;
        const uint32_t na = (nd ^ (A * 7u)) - A * (uint32_t)(7 - 2 * D);
        bond += 8 * D - 2 * (long long)__dp4a(na, ones, 0u);
        down += (long long)__dp4a(A, ones, __dp4a(cur, ones, 0u));
    };
    if ((Q & 3) == 0) {
        // 16-byte chunks of four words: 128-bit loads, the x shift inside the
        // chunk, one edge word from the chunk beside it
        const int Q4 = Q >> 2;
        const uint4* own4 = reinterpret_cast<const uint4*>(own);
        const uint4* oth4 = reinterpret_cast<const uint4*>(oth);
        const RowSplit rs(Q4);
        for (long long row = (long long)blockIdx.x * rs.rpb + rs.rsub;
             rs.rsub < rs.rpb && row < rows; row += (long long)gridDim.x * rs.rpb) {
            const int y = (int)(row % L), z = D == 3 ? (int)(row / L) : 0;
            const int p = (y + z + 1) & 1;
            const long long ym = row - y + (y == 0 ? L - 1 : y - 1);
            const long long yp = row - y + (y == L - 1 ? 0 : y + 1);
            const long long zm = D == 3 ? ((z == 0 ? L - 1 : z - 1) * (long long)L + y) : 0;
            const long long zp = D == 3 ? ((z == L - 1 ? 0 : z + 1) * (long long)L + y) : 0;
            for (int c = rs.q0; c < Q4; c += rs.tq) {
                const uint4 A = __ldcs(own4 + row * Q4 + c);
                const uint4 cur = __ldg(oth4 + row * Q4 + c);
                const uint32_t edge =
                    __ldg(oth + row * Q + (p ? (c + 1 == Q4 ? 0 : 4 * c + 4) : (c == 0 ? Q - 1 : 4 * c - 1)));
                uint4 nv = __ldg(oth4 + ym * Q4 + c);
                const uint4 v2 = __ldg(oth4 + yp * Q4 + c);
                nv.x += v2.x;
                nv.y += v2.y;
                nv.z += v2.z;
                nv.w += v2.w;
                if (D == 3) {
                    const uint4 v3 = __ldg(oth4 + zm * Q4 + c);
                    const uint4 v4 = __ldg(oth4 + zp * Q4 + c);
                    nv.x += v3.x + v4.x;
                    nv.y += v3.y + v4.y;
                    nv.z += v3.z + v4.z;
                    nv.w += v3.w + v4.w;
                }
                if (p) {
                    word(A.x, cur.x, __funnelshift_r(cur.x, cur.y, 8), nv.x);
                    word(A.y, cur.y, __funnelshift_r(cur.y, cur.z, 8), nv.y);
                    word(A.z, cur.z, __funnelshift_r(cur.z, cur.w, 8), nv.z);
                    word(A.w, cur.w, __funnelshift_r(cur.w, edge, 8), nv.w);
                } else {
                    word(A.x, cur.x, __funnelshift_l(edge, cur.x, 8), nv.x);
                    word(A.y, cur.y, __funnelshift_l(cur.x, cur.y, 8), nv.y);
                    word(A.z, cur.z, __funnelshift_l(cur.y, cur.z, 8), nv.z);
                    word(A.w, cur.w, __funnelshift_l(cur.z, cur.w, 8), nv.w);
                }
            }
        }
    }
    const RowSplit rs(Q);
    for (long long row = (long long)blockIdx.x * rs.rpb + rs.rsub;
         (Q & 3) != 0 && rs.rsub < rs.rpb && row < rows; row += (long long)gridDim.x * rs.rpb) {
        const int y = (int)(row % L), z = D == 3 ? (int)(row / L) : 0;
        const int p = (y + z + 1) & 1;
        const long long base = row * Q;
        for (int q = rs.q0; q < Q; q += rs.tq) {
            const uint32_t A = __ldcs(own + base + q);
            const uint32_t cur = __ldg(oth + base + q);
            const uint32_t S =
                p ? __funnelshift_r(cur, __ldg(oth + base + (q + 1 == Q ? 0 : q + 1)), 8)
                  : __funnelshift_l(__ldg(oth + base + (q == 0 ? Q - 1 : q - 1)), cur, 8);
            const long long ym = row - y + (y == 0 ? L - 1 : y - 1);
            const long long yp = row - y + (y == L - 1 ? 0 : y + 1);
            uint32_t nv = __ldg(oth + ym * Q + q) + __ldg(oth + yp * Q + q);
            if (D == 3) {
                const long long zm = (z == 0 ? L - 1 : z - 1), zp = (z == L - 1 ? 0 : z + 1);
                nv += __ldg(oth + (zm * L + y) * Q + q) + __ldg(oth + (zp * L + y) * Q + q);
            }
            word(A, cur, S, nv);
        }
    }
    Partial mine;
    mine.i0 = block_sum(bond, red);
    mine.i1 = block_sum(down, red);
    mine.f[0] = mine.f[1] = mine.f[2] = mine.f[3] = 0.0;
    finish_pass<false>(a.ctrl, partials, mine, [&](const Partial& tot) {
        Ctrl* C = a.ctrl;
        const double E = -J * (double)tot.i0;
        const double M = (double)(a.N - 2 * tot.i1);
        C->obs[0] = E;
        C->obs[1] = M;
        C->obs[2] = 0.0;
        C->obs[3] = 0.0;
        const long long k = series_place(C, C->t);
        if (C->series_E) C->series_E[k] = E;
        if (C->series_absm) C->series_absm[k] = fabs(M) / (double)a.N;
        C->t = C->t + 1;
    });
}

template <int D>
long long tiles_of(int L, int& ntx, int& nty, int& ntz)
{
    ntx = (L + SwTile<D>::TX - 1) / SwTile<D>::TX;
    nty = (L + SwTile<D>::TY - 1) / SwTile<D>::TY;
    ntz = D == 3 ? (L + SwTile<D>::TZ - 1) / SwTile<D>::TZ : 1;
    return (long long)ntx * nty * ntz;
}

template <int D>
cudaError_t sw_update(const SwArgs& a0, cudaStream_t s)
{
    SwArgs a = a0;
    const long long mergers = a.ntiles * SwFace<D>::WORDS * 32;
    cudaError_t e = cudaMemsetAsync(a.nroots, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    const dim3 tiles((unsigned)a.ntx, (unsigned)a.nty, (unsigned)a.ntz);
    if (D == 2) sw_local2<<<tiles, kSwThreads2, 0, s>>>(a);
    else sw_local3<<<tiles, kSwThreads, 0, s>>>(a);
    sw_merge<D><<<grid_for(mergers, 256), 256, 0, s>>>(a);
    sw_resolve<<<grid_for(a.N, 256), 256, 0, s>>>(a);
    sw_flip<<<grid_for((a.N / 2 + 3) / 4, 256), 256, 0, s>>>(a);  // at most one block per row used
    return cudaGetLastError();
}

}  // namespace

size_t sw_workspace_bytes(int d, int L)
{
    int ntx, nty, ntz;
    const size_t N = (size_t)L * L * (d == 3 ? L : 1);
    const long long nt = d == 2 ? tiles_of<2>(L, ntx, nty, ntz) : tiles_of<3>(L, ntx, nty, ntz);
    const size_t words = d == 2 ? SwFace<2>::WORDS : SwFace<3>::WORDS;
    // labels, tile-face bits, the tile-root list and its count
    return align_up(N * 4) + align_up((size_t)nt * words * 4) + align_up(N * 4) + align_up(4);
}

cudaError_t ising_sw_sweeps(const sl_lattice* h, const SweepParams& p, int64_t count,
                            cudaStream_t s)
{
    SwArgs a;
    a.s[0] = (int8_t*)h->spins[0];
    a.s[1] = (int8_t*)h->spins[1];
    a.lab = (uint32_t*)h->ws;
    a.face = (uint32_t*)((char*)h->ws + align_up((size_t)h->N * 4));
    {
        int ntx, nty, ntz;
        const long long nt = h->d == 2 ? tiles_of<2>(h->L, ntx, nty, ntz)
                                       : tiles_of<3>(h->L, ntx, nty, ntz);
        const size_t words = h->d == 2 ? SwFace<2>::WORDS : SwFace<3>::WORDS;
        char* after_face = (char*)a.face + align_up((size_t)nt * words * 4);
        a.roots = (uint32_t*)after_face;
        a.nroots = (unsigned*)(after_face + align_up((size_t)h->N * 4));
    }
    a.L = h->L;
    a.N = h->N;
    a.ntiles = h->d == 2 ? tiles_of<2>(h->L, a.ntx, a.nty, a.ntz)
                         : tiles_of<3>(h->L, a.ntx, a.nty, a.ntz);
    a.ntxd = make_fast_div((uint32_t)a.ntx);
    a.ntyd = make_fast_div((uint32_t)a.nty);
    a.thr = p.tab.sw_thr;
    a.never = p.tab.sw_never;
    a.anti = h->J < 0.0;
    a.replica = h->replica;
    a.rk = p.rk;
    a.ctrl = h->ctrl;
    for (int64_t k = 0; k < count; ++k) {
        cudaError_t e = h->d == 2 ? sw_update<2>(a, s) : sw_update<3>(a, s);
        if (e == cudaSuccess) {
            if (h->L % 8 == 0) {
                const long long items = (long long)h->L * (h->d == 3 ? h->L : 1) * (h->L / 8);
                int grid = grid_for(items, 256);
                if (grid > kI8Blocks) grid = kI8Blocks;
                if (h->d == 2) sw_measure<2><<<grid, 256, 0, s>>>(a, h->partials, h->J);
                else sw_measure<3><<<grid, 256, 0, s>>>(a, h->partials, h->J);
                e = cudaGetLastError();
            } else {
                e = ising_i8_measure_advance(h, s);
            }
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace spinmc
