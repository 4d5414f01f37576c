// xy_ccl.cu -- labelling of frozen domains after a quench (paper: frozen
// domains and their size distribution, abstract and Fig. 6; Sec. IV.C).
//
// A site's Ising projection is spin = (theta >= 0), the sign of
// s = sin(2 theta) on [-pi/2, pi/2) (Sec. IV.A).  Domains are the connected
// components of equal spin under 4-neighbour adjacency with periodic wrap.
// Each site gets the smallest site index of its component, which makes the
// labels unique and comparable bit for bit.
//
// Passes (unions always link the larger root under the smaller, so every
// root is its component's minimum):
//   tile    one warp per 32 x 32 tile: the rows' spins as 32-bit masks, runs
//           of equal spin, each linked to one run of the row above, pointer
//           jumping, and unions in shared memory for the remaining contacts;
//           every site gets its tile root, and each piece its tile-local size.
//           A piece that does not reach the tile's edge is a whole domain and
//           goes into the size histogram at once; one that does goes on a
//           short list (batch index, local size) for the merge.
//   border  one warp per tile, from the spins and tile roots of the edge sites
//           that the tile pass kept: one union in global memory per pair of
//           runs that touch across the tile's right and bottom edges.
//   sizes   the listed pieces add their local sizes at their domain's root's
//           entry of the list (and point their tile roots at the root); the
//           roots' entries then enter the histogram.
//   flatten one warp per tile: every site points straight at its root.
//   compact the histogram's nonzero entries become (size, count) pairs in
//           ascending order: sizes below 64 are summed over the copies their
//           counts are spread over, larger ones are found through a bitmap
//           with one bit per size.
// The histogram counts, their copies and the bitmap are zero between calls:
// the passes clear every entry they set, so no pass reads or clears memory in
// proportion to the lattice beyond the labels themselves.
#include <algorithm>
#include <cstdint>

#include "xy_internal.h"

namespace xy {

namespace {

constexpr int kMaxUnionIters = 1 << 22;
constexpr unsigned kAll = 0xFFFFFFFFu;
constexpr int kTileWarps = 4;      // tiles (warps) per block of the tile pass
constexpr int kSmallSizes = 64;    // sizes counted in shared memory before the global histogram
constexpr int kEdgeFlag = 1 << 16;  // added to a piece's size count for each of its runs on the tile edge

}  // namespace

// Upper bound on the steps of one root search and on the link retries of one
// union in global memory (per device).  xy_debug_set_union_limit() lowers it
// so that tests can run the timeout path: a loop that reaches the bound sets
// XY_ETIMEOUT and returns, and since links only ever point at smaller
// indices the forest stays acyclic and every index stays in range.
__device__ int g_union_limit = kMaxUnionIters;

namespace {

__device__ __forceinline__ bool spin_of(float t) { return t >= 0.0f; }

// Bit x set where a run of equal bits starts in the row mask m (bit 0 always),
// over the tile's columns vm.
__device__ __forceinline__ unsigned run_starts(unsigned m, unsigned vm) { return ((m ^ (m << 1)) | 1u) & vm; }

// Column of the start of the run that holds column x.
__device__ __forceinline__ int run_of(unsigned starts, int x) { return 31 - __clz(starts & ((2u << x) - 1u)); }

// Root of x in the forest L (global memory), halving the path on the way:
// each visited node is pointed at its grandparent, an ancestor, so concurrent
// searches and links stay valid.
__device__ __forceinline__ int find_root_global(int32_t* L, int x, int limit, int* err)
{
    int p = *(volatile const int32_t*)&L[x];
    for (int it = 0; p != x; ++it) {
        if (it >= limit) {
            atomicExch(err, XY_ETIMEOUT);
            return x;
        }
        const int g = *(volatile const int32_t*)&L[p];
        if (g == p) return p;
        L[x] = g;
        x = g;
        p = *(volatile const int32_t*)&L[x];
    }
    return x;
}

// The same search without writes (used while the owners of nodes point them
// at their roots: a halving step could replace such a pointer with an older
// ancestor).
__device__ __forceinline__ int find_root_global_ro(const int32_t* L, int x, int limit, int* err)
{
    int p = *(volatile const int32_t*)&L[x];
    for (int it = 0; p != x; ++it) {
        if (it >= limit) {
            atomicExch(err, XY_ETIMEOUT);
            return x;
        }
        x = p;
        p = *(volatile const int32_t*)&L[x];
    }
    return x;
}

// Link the components of a and b (global indices inside one lattice's label
// array L): the larger root is pointed at the smaller with atomicMin; a failed
// link (the root changed meanwhile) retries from the value it found.
__device__ void union_global(int32_t* L, int a, int b, int limit, int* err)
{
    for (int it = 0; it < limit; ++it) {
        a = find_root_global(L, a, limit, err);
        b = find_root_global(L, b, limit, err);
        if (a == b) return;
        if (a < b) {
            const int t = a;
            a = b;
            b = t;
        }
        const int old = atomicMin(&L[a], b);
        if (old == a) return;
        a = old;
    }
    atomicExch(err, XY_ETIMEOUT);
}

// Tile-local site i = y * 32 + x lives at shared-memory word i + y (rows
// padded to 33 words): lanes that each own a row and touch the same column
// then hit 32 different banks.  Indices keep the site order; only the
// address is padded.
__device__ __forceinline__ int ph(int i) { return i + (i >> 5); }

// Root of x in a tile's forest (padded layout), halving the path.
__device__ __forceinline__ int find_root_tile(int* L, int x)
{
    int p = L[ph(x)];
    while (p != x) {
        const int g = L[ph(p)];
        if (g == p) return p;
        L[ph(x)] = g;
        x = g;
        p = L[ph(x)];
    }
    return x;
}

// Link in a tile's forest (padded layout), with a bound on the retries:
// every failed atomicMin means another lane lowered the same entry, so the
// loop ends long before the bound in practice; reaching it sets XY_ETIMEOUT
// like the global loops (the forest stays valid, links only point at
// smaller indices).
__device__ void union_tile(int* L, int a, int b, int* err)
{
    for (int it = 0; it < 4096 * 4; ++it) {
        a = find_root_tile(L, a);
        b = find_root_tile(L, b);
        if (a == b) return;
        if (a < b) {
            const int t = a;
            a = b;
            b = t;
        }
        const int old = atomicMin(&L[ph(a)], b);
        if (old == a) return;
        a = old;
    }
    atomicExch(err, XY_ETIMEOUT);
}

// how_many more domains of size sz in lattice lat's histogram.  Small sizes
// are hot (every tile has some): their counts are spread over s.copies
// copies per lattice, picked by tile, and the compaction adds the copies.  A
// larger size is marked in the bitmap by the first add that finds its count
// at zero, so no lane reads a shared word.
__device__ __forceinline__ void count_size(const CclScratch& s, int64_t N, int lat, int sz, int how_many, int tile)
{
    if (sz < kSmallSizes) {
        atomicAdd(s.small + ((int64_t)lat * s.copies + tile % s.copies) * kSmallSizes + sz, how_many);
    } else if (atomicAdd(s.counts + (int64_t)lat * (N + 1) + sz, how_many) == 0) {
        atomicOr(s.bits + (int64_t)lat * s.words + (sz >> 5), 1u << (sz & 31));
    }
}

// Shared memory of one tile: the forest over run starts (tile-local index
// y * 32 + x at word ph(i); other entries unused), and the counts of small
// sizes.  Once the forest is final, a root's own entry holds
// -1 - (size + kEdgeFlag * edge runs) of its piece: every other run start
// then points straight at its root, so the entry is free.
struct TileSmem {
    int P[32 * 33];
    int H[kSmallSizes];
};

}  // namespace

// Pass 1: one warp per tile of up to 32 x 32 sites (the last tile of a row or
// column of tiles may be narrower).  Tile-local indices y * 32 + x order like
// global indices, so a tile root is its piece's smallest site.
__global__ void __launch_bounds__(32 * kTileWarps, 12) ccl_tile_kernel(const float* __restrict__ theta, int Lx, int Ly,
                                                                     int n_lat, int32_t* __restrict__ labels,
                                                                     CclScratch s, int* err)
{
    __shared__ TileSmem sm[kTileWarps];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int tiles_x = (Lx + 31) >> 5, tiles_y = (Ly + 31) >> 5;
    const int tiles = tiles_x * tiles_y;  // the batch has fewer than 2^31 sites
    const int t = blockIdx.x * kTileWarps + wib;
    if (t >= tiles * n_lat) return;  // a whole warp
    const int lat = t / tiles;
    const int tile = t - lat * tiles;
    const int ty = tile / tiles_x, tx = tile - ty * tiles_x;
    const int gx0 = tx * 32, gy0 = ty * 32;
    const int tw = min(32, Lx - gx0), thh = min(32, Ly - gy0);
    const unsigned vm = tw == 32 ? kAll : ((1u << tw) - 1u);
    const int64_t N = (int64_t)Lx * Ly;
    const float* th = theta + (int64_t)lat * N + gy0 * Lx + gx0;
    int32_t* lab = labels + (int64_t)lat * N + gy0 * Lx + gx0;
    int* P = sm[wib].P;
    int* H = sm[wib].H;

    // the rows' spins as masks (lane y keeps row y); 16 loads in flight per lane
    unsigned row = 0;
    if (tw == 32 && thh == 32) {
#pragma unroll
        for (int h = 0; h < 32; h += 16) {
            float v[16];
#pragma unroll
            for (int y = 0; y < 16; ++y) v[y] = th[(h + y) * Lx + lane];
#pragma unroll
            for (int y = 0; y < 16; ++y) {
                const unsigned m = __ballot_sync(kAll, spin_of(v[y]));
                row = lane == h + y ? m : row;
            }
        }
    } else {
        for (int y = 0; y < thh; ++y) {
            const unsigned m = __ballot_sync(kAll, spin_of(lane < tw ? th[y * Lx + lane] : 0.0f)) & vm;
            row = lane == y ? m : row;
        }
    }
    const unsigned st = lane < thh ? run_starts(row, vm) : 0u;  // lane y: the run starts of row y

    // Every run is linked to the first run it touches in the row above (a smaller
    // index), or is a root: each lane writes only its own run starts, so the tree
    // needs no search and no atomic.  Its other contacts with the row above (at the
    // first column where a pair of runs touches) are left in `more`: they join two
    // pieces, or close a loop.
    unsigned more = 0, sa;
    {
        const unsigned above = __shfl_up_sync(kAll, row, 1);
        sa = __shfl_up_sync(kAll, st, 1);
        const unsigned c = lane > 0 && lane < thh ? ~(row ^ above) & vm : 0u;
        const unsigned u = c & ~((c << 1) & c & ~st & ~sa);
        for (unsigned b = st; b; b &= b - 1) {
            const unsigned later = b & (b - 1);
            const int x = __ffs(b) - 1;
            // contacts of this run: from its start up to the next one
            const unsigned uu = u & (later ? (later & (0u - later)) - 1u : kAll) & (kAll << x);
            P[lane * 33 + x] = uu ? lane * 32 - 32 + run_of(sa, __ffs(uu) - 1) : lane * 32 + x;
            more |= uu & (uu - 1);
        }
    }
    H[lane] = 0;
    H[lane + 32] = 0;
    __syncwarp();
    // Pointer jumping: every run start points at its grandparent until all point
    // at roots, log2 of the longest chain passes (a lane writes only its own
    // entries, and only ancestors, so the passes need no order among the lanes).
    // A search from each run start walked chains of up to 32 rows instead.
    volatile int* vP = P;
    auto jump = [&]() {
        for (int pass = 0; pass < 33; ++pass) {
            bool moved = false;
            for (unsigned b = st; b; b &= b - 1) {
                const int i = lane * 33 + __ffs(b) - 1;
                const int p = vP[i];
                const int g = vP[ph(p)];
                if (g != p) {
                    vP[i] = g;
                    moved = true;
                }
            }
            __syncwarp();
            if (!__any_sync(kAll, moved)) break;
        }
    };
    jump();
    if (__any_sync(kAll, more != 0u)) {
        for (unsigned b = more; b; b &= b - 1) {
            const int x = __ffs(b) - 1;
            union_tile(P, lane * 32 + run_of(st, x), lane * 32 - 32 + run_of(sa, x), err);
        }
        __syncwarp();
        jump();
    }

    unsigned roots = 0;  // lane y: the tile roots of row y
    for (unsigned b = st; b; b &= b - 1) {
        const int x = __ffs(b) - 1;
        if (P[lane * 33 + x] == lane * 32 + x) roots |= b & (0u - b);
    }
    // (a tile whose unions ran out of retries still has every root in `roots`)
    __syncwarp();
    // a root's entry becomes its piece's count: -1 - (size + kEdgeFlag * edge runs)
    for (unsigned b = roots; b; b &= b - 1) P[lane * 33 + __ffs(b) - 1] = -1;
    __syncwarp();
    for (unsigned b = st; b; b &= b - 1) {
        const int x = __ffs(b) - 1;
        const int i = lane * 32 + x;
        const int q = P[lane * 33 + x];
        const int r = q < 0 ? i : q;
        const unsigned later = b & (b - 1);
        const int end = later ? __ffs(later) - 1 : tw;
        const bool edge = lane == 0 || lane == thh - 1 || x == 0 || end == tw;
        atomicSub(&P[ph(r)], (end - x) + (edge ? kEdgeFlag : 0));
    }
    __syncwarp();

    // the tile roots and spins of the edge sites go to the border pass: top row,
    // bottom row (lane = column), left column, right column (lane = row)
    {
        uint16_t* er = s.edge_root + (int64_t)t * 128;
        auto root_at = [&](int y, int x) {  // of the run that starts at (x, y)
            const int q = P[y * 33 + x];
            return (uint16_t)(q < 0 ? y * 32 + x : q);
        };
        const unsigned st_top = __shfl_sync(kAll, st, 0), st_bottom = __shfl_sync(kAll, st, thh - 1);
        if (lane < tw) {
            er[lane] = root_at(0, run_of(st_top, lane));
            er[32 + lane] = root_at(thh - 1, run_of(st_bottom, lane));
        }
        if (lane < thh) {
            er[64 + lane] = root_at(lane, 0);
            er[96 + lane] = root_at(lane, run_of(st, tw - 1));
        }
        const unsigned left = __ballot_sync(kAll, lane < thh && (row & 1u));
        const unsigned right = __ballot_sync(kAll, lane < thh && ((row >> (tw - 1)) & 1u));
        const unsigned top = __shfl_sync(kAll, row, 0), bottom = __shfl_sync(kAll, row, thh - 1);
        if (lane == 0) s.edge_spin[t] = make_uint4(top, bottom, left, right);
    }

    // the pieces: whole domains into the histogram, edge pieces onto the list
    int n_edge = 0;
    for (unsigned b = roots; b; b &= b - 1) n_edge += -1 - P[lane * 33 + __ffs(b) - 1] >= kEdgeFlag;
    int before = n_edge;  // inclusive prefix over the lanes
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(kAll, before, d);
        if (lane >= d) before += o;
    }
    const int total = __shfl_sync(kAll, before, 31);
    int base = 0;
    if (lane == 31 && total > 0) base = atomicAdd(s.list_n, total);
    base = __shfl_sync(kAll, base, 31) + before - n_edge;
    for (unsigned b = roots; b; b &= b - 1) {
        const int x = __ffs(b) - 1;
        const int c = -1 - P[lane * 33 + x];
        const int sz = c & (kEdgeFlag - 1);
        if (c >= kEdgeFlag) {
            if (base < s.list_cap) {
                const int g = (gy0 + lane) * Lx + gx0 + x;
                s.list[base] = make_int2((int)((int64_t)lat * N + g), sz);
                s.aux[base] = make_int2(-1, 0);
                s.entry[(int64_t)lat * N + g] = base;
            } else {
                atomicExch(err, XY_ENOMEM);  // not reached: the capacity bounds the pieces on tile edges
            }
            ++base;
        } else if (sz < kSmallSizes) {
            atomicAdd(&H[sz], 1);
        } else {
            count_size(s, N, lat, sz, 1, tile);
        }
    }
    __syncwarp();
    // labels: every run start's entry becomes its root's site in the lattice (each
    // lane its own entries), then a row at a time (coalesced), each site through
    // its run start
    for (unsigned b = st; b; b &= b - 1) {
        const int x = __ffs(b) - 1;
        const int q = P[lane * 33 + x];
        const int r = q < 0 ? lane * 32 + x : q;
        P[lane * 33 + x] = (gy0 + (r >> 5)) * Lx + gx0 + (r & 31);
    }
    P[lane * 33 + 32] = (int)st;  // (the padding word of each row)
    __syncwarp();
    if (lane < tw) {
        const unsigned upto = (2u << lane) - 1u;
        int32_t* o = lab + lane;
#pragma unroll 8
        for (int y = 0; y < thh; ++y) {
            *o = P[y * 33 + 31 - __clz((unsigned)P[y * 33 + 32] & upto)];
            o += Lx;
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int sz = lane + 32 * k;
        if (H[sz] > 0) count_size(s, N, lat, sz, H[sz], tile);
    }
}

// Pass 2: merge across the right and bottom edge of every tile (periodic).
// One warp per tile; lane k takes the k-th site of the right edge (against
// the first column of the next tile) and of the bottom edge (against the top
// row of the tile below).  The spins and tile roots of edge sites come from
// the tile pass (no angle or label is read along the edges).  Where the
// previous lane also touches and its site continues the run along the edge
// (then so does the neighbour's, which has the same spin), the pair of
// pieces is already linked: one union per pair of touching runs.  The roots'
// entries are read at once for both edges; two roots are then linked
// straight away, anything else goes through the general union.
// Its threads also clear the histogram's pairs (hist, n_hist words; the compaction
// fills the leading ones): one block per lattice spent longer on that than on the
// pairs.
__global__ void __launch_bounds__(256) ccl_border_kernel(int Lx, int Ly, int n_lat, int32_t* labels, CclScratch s,
                                                         int64_t* hist, int64_t n_hist, int* err)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_hist; i += (int64_t)gridDim.x * blockDim.x)
        hist[i] = 0;
    const int lane = threadIdx.x & 31;
    const int tiles_x = (Lx + 31) >> 5, tiles_y = (Ly + 31) >> 5;
    const int tiles = tiles_x * tiles_y;
    const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t >= tiles * n_lat) return;  // a whole warp
    const int lat = t / tiles;
    const int tile = t - lat * tiles;
    const int ty = tile / tiles_x, tx = tile - ty * tiles_x;
    const int gx0 = tx * 32, gy0 = ty * 32;
    const int tw = min(32, Lx - gx0), thh = min(32, Ly - gy0);
    const int txr = tx + 1 == tiles_x ? 0 : tx + 1, tyb = ty + 1 == tiles_y ? 0 : ty + 1;
    const int t0 = lat * tiles;
    const int tr = t0 + ty * tiles_x + txr, tb = t0 + tyb * tiles_x + tx;  // the tiles to the right and below
    int32_t* L = labels + (int64_t)lat * Lx * Ly;
    const int limit = g_union_limit;
    const uint4 me = s.edge_spin[t];
    const unsigned sp_right = me.w, sp_bottom = me.y;
    const unsigned sp_nleft = s.edge_spin[tr].z, sp_ntop = s.edge_spin[tb].x;
    const uint16_t* er = s.edge_root + (int64_t)t * 128;
    // edge 0: right (rows k < thh); edge 1: bottom (columns k < tw)
    int a[2], b[2];
    bool need[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const bool act = lane < (e == 0 ? thh : tw);
        const unsigned ms = e == 0 ? sp_right : sp_bottom, mn = e == 0 ? sp_nleft : sp_ntop;
        const bool sa = act && ((ms >> lane) & 1u);
        const bool touch = act && sa == (((mn >> lane) & 1u) != 0);
        const unsigned tm = __ballot_sync(kAll, touch);
        const bool prev_sa = __shfl_up_sync(kAll, sa, 1);
        need[e] = touch && !(lane > 0 && ((tm >> (lane - 1)) & 1u) && prev_sa == sa);
        a[e] = b[e] = 0;
        if (need[e]) {
            const int ra = er[(e == 0 ? 96 : 32) + lane];
            const int rb = s.edge_root[(int64_t)(e == 0 ? tr : tb) * 128 + (e == 0 ? 64 : 0) + lane];
            const int gxn = e == 0 ? txr * 32 : gx0, gyn = e == 0 ? gy0 : tyb * 32;
            a[e] = (gy0 + (ra >> 5)) * Lx + gx0 + (ra & 31);
            b[e] = (gyn + (rb >> 5)) * Lx + gxn + (rb & 31);
        }
    }
    int pa[2], pb[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        pa[e] = need[e] ? L[a[e]] : 0;
        pb[e] = need[e] ? L[b[e]] : 0;
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        if (!need[e]) continue;
        if (pa[e] == a[e] && pb[e] == b[e]) {  // two roots
            if (a[e] == b[e]) continue;
            const int hi = max(a[e], b[e]), lo = min(a[e], b[e]);
            const int old = atomicMin(&L[hi], lo);
            if (old != hi) union_global(L, old, lo, limit, err);  // hi was linked meanwhile
        } else {
            union_global(L, a[e], b[e], limit, err);
        }
    }
}

// Pass 3: each listed piece finds its domain's root, points its tile root
// there, and adds its tile-local size to the root's own entry of the list
// (the root is the tile root of a listed piece: a domain that spans tiles
// reaches the edge of each of its tiles; the tile pass recorded each listed
// tile root's entry).  Searches write nothing here, so afterwards every tile
// root of a merged piece points straight at its domain's root.  A block
// takes 256 consecutive entries from a few tiles; a domain spanning many
// tiles would get an atomic from nearly every entry, all on one address, so
// the pieces of the block's first entry's domain are summed in shared
// memory and added once.
__global__ void __launch_bounds__(256) ccl_list_size_kernel(int64_t N, int32_t* labels, CclScratch s, int* err)
{
    __shared__ int s_key;
    __shared__ int s_sum;
    const int n = min(*s.list_n, (int)s.list_cap);
    const int limit = g_union_limit;
    for (int base = blockIdx.x * blockDim.x; base < n; base += gridDim.x * blockDim.x) {
        const int i = base + threadIdx.x;
        int key = -1, sz = 0;
        if (i < n) {
            const int2 e = s.list[i];
            const int lat = (int)(e.x / N);
            const int g = (int)(e.x - lat * N);
            int32_t* L = labels + (int64_t)lat * N;
            const int r = find_root_global_ro(L, g, limit, err);
            if (r != g) L[g] = r;  // every merged tile root now points at its domain's root
            key = r == g ? i : s.entry[(int64_t)lat * N + r];
            // the root's entry, checked (a search cut short by the bound ends
            // at a node that may not be listed)
            if (key < 0 || key >= n || s.list[key].x != (int)((int64_t)lat * N + r)) {
                atomicExch(err, XY_ETIMEOUT);
                key = -1;
            }
            s.aux[i].x = key;
            sz = e.y;
        }
        if (threadIdx.x == 0) {
            s_key = key;
            s_sum = 0;
        }
        __syncthreads();
        const int k0 = s_key;
        if (key >= 0) {
            if (key == k0)
                atomicAdd(&s_sum, sz);
            else
                atomicAdd(&s.aux[key].y, sz);
        }
        __syncthreads();
        if (threadIdx.x == 0 && s_sum > 0) atomicAdd(&s.aux[k0].y, s_sum);
        __syncthreads();
    }
}

// Pass 3b: the listed pieces whose tile root is their domain's root enter the
// histogram with the domain's size.  A block takes 256 consecutive entries,
// from a few tiles of one lattice: small sizes of that lattice are counted
// in shared memory and added with one atomic per size.
__global__ void __launch_bounds__(256) ccl_list_hist_kernel(int64_t N, CclScratch s, int* err)
{
    __shared__ int bins[kSmallSizes];
    __shared__ int blat;
    const int n = min(*s.list_n, (int)s.list_cap);
    for (int base = blockIdx.x * blockDim.x; base < n; base += gridDim.x * blockDim.x) {
        if (threadIdx.x < kSmallSizes) bins[threadIdx.x] = 0;
        if (threadIdx.x == 0) blat = (int)(s.list[base].x / N);
        __syncthreads();
        const int i = base + threadIdx.x;
        if (i < n) {
            const int2 a = s.aux[i];
            if (a.x == i && (a.y < 1 || a.y > N)) {
                atomicExch(err, XY_ETIMEOUT);  // only after a search was cut short
            } else if (a.x == i) {
                const int l = (int)(s.list[i].x / N);
                if (l == blat && a.y < kSmallSizes)
                    atomicAdd(&bins[a.y], 1);
                else
                    count_size(s, N, l, a.y, 1, blockIdx.x);
            }
        }
        __syncthreads();
        if (threadIdx.x < kSmallSizes && bins[threadIdx.x] > 0)
            count_size(s, N, blat, threadIdx.x, bins[threadIdx.x], blockIdx.x);
        __syncthreads();
    }
}

// Pass 4: every site points straight at its root; one warp per tile, lane =
// column.  A site's label is its tile root, a site of the same tile (the
// tile root's own entry is the exception: after a merge it points outside),
// and after pass 3 the tile root's own entry is the domain's root (or
// itself): so the warp reads the tile's labels once (16 rows at a time per
// lane), keeps them in shared memory, and looks every tile root up there.  A
// site whose tile root is still a root is final and is not written.
// A width that is a power of two (shift >= 0) gives a label's row and column by a
// shift and a mask; others by a product and a correction.
template <bool POW2>
__global__ void __launch_bounds__(256, 4) ccl_flatten_kernel(int Lx, int Ly, int n_lat, float inv_lx, int shift,
                                                             int32_t* labels)
{
    __shared__ int T[8][32 * 33];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int tiles_x = (Lx + 31) >> 5, tiles_y = (Ly + 31) >> 5;
    const int tiles = tiles_x * tiles_y;
    const int t = blockIdx.x * 8 + wib;
    if (t >= tiles * n_lat) return;  // a whole warp
    const int lat = t / tiles;
    const int tile = t - lat * tiles;
    const int ty = tile / tiles_x, tx = tile - ty * tiles_x;
    const int gx0 = tx * 32, gy0 = ty * 32;
    const int tw = min(32, Lx - gx0), thh = min(32, Ly - gy0);
    const bool in = lane < tw;
    int32_t* L = labels + (int64_t)lat * Lx * Ly;
    const int base = gy0 * Lx + gx0;
    int* Tw = T[wib];
#pragma unroll
    for (int h = 0; h < 32; h += 16) {
        int l[16];
#pragma unroll
        for (int y = 0; y < 16; ++y) l[y] = (in && h + y < thh) ? L[base + (h + y) * Lx + lane] : 0;
#pragma unroll
        for (int y = 0; y < 16; ++y) Tw[(h + y) * 33 + lane] = l[y];
    }
    __syncwarp();
    if (!in) return;
#pragma unroll 4
    for (int y = 0; y < thh; ++y) {
        const int li = Tw[y * 33 + lane];
        const int d = li - base;  // a site of the tile at row ry, column rx: d = ry * Lx + rx
        int ry, rx;
        if (POW2) {
            ry = d >> shift;
            rx = d & (Lx - 1);
        } else {
            ry = (int)((float)d * inv_lx);
            if (ry * Lx > d)
                --ry;
            else if ((ry + 1) * Lx <= d)
                ++ry;
            rx = d - ry * Lx;
        }
        // a label outside the tile belongs to a tile root whose entry points
        // at its domain's root already: final
        if ((unsigned)ry < (unsigned)thh && (unsigned)rx < (unsigned)tw) {
            const int p = Tw[ry * 33 + rx];
            if (p != li) L[base + y * Lx + lane] = p;
        }
    }
}

constexpr int kWordList = 1024;

// Pass 5: ordered compaction of the nonzero counts into (size, count) pairs,
// one block per lattice, ascending size (the rest of the lattice's hist_cap
// pairs is zero already).  Sizes 1..63 are summed over their copies; larger ones
// are found through the bitmap, one bit per size: a warp takes 1024 consecutive
// words, all 32 loads of a lane in flight, the warps' bits are summed in one
// block-wide prefix, and the words that hold any go onto a list that all warps
// share, a lane per size: a lane that walked a dense word waited for one count
// after the other, and a round of 1024 words at a time took four barriers.
__global__ void __launch_bounds__(1024, 1) ccl_compact_kernel(int64_t N, CclScratch s, int64_t* hist, int64_t hist_cap,
                                                           int64_t* n_sizes, int* err)
{
    __shared__ int s_warp[32];
    __shared__ int s_small[kSmallSizes];
    __shared__ uint4 s_list[kWordList];  // word index, word, position of its first pair
    __shared__ int s_n;
    const int lat = blockIdx.x;
    int32_t* cnt = s.counts + (int64_t)lat * (N + 1);
    uint32_t* bw = s.bits + (int64_t)lat * s.words;
    int64_t* out = hist ? hist + (int64_t)lat * hist_cap * 2 : nullptr;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    const int n_small = (int)(N < kSmallSizes - 1 ? N : kSmallSizes - 1);  // sizes 1..n_small
    if (threadIdx.x < kSmallSizes) s_small[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    {
        // thread j adds copies j / 64, j / 64 + 16, ... of size j % 64: every
        // copy is read by one thread, at most two loads deep
        const int z = threadIdx.x & (kSmallSizes - 1);
        const int nk = (int)blockDim.x / kSmallSizes;
        int v = 0;
        if (z >= 1 && z <= n_small) {
            for (int k = (int)threadIdx.x / kSmallSizes; k < s.copies; k += nk) {
                int32_t* c = s.small + ((int64_t)lat * s.copies + k) * kSmallSizes + z;
                const int a = *c;
                if (a) {
                    v += a;
                    *c = 0;
                }
            }
        }
        if (v) atomicAdd(&s_small[z], v);
    }
    __syncthreads();
    int64_t pos = 0;  // pairs placed so far (the same in every thread)
#pragma unroll
    for (int k = 0; k < kSmallSizes / 32; ++k) {
        const int z = lane + 32 * k;
        const unsigned m = __ballot_sync(kAll, s_small[z] != 0);
        const int64_t at = pos + __popc(m & below);
        if (warp == 0 && s_small[z] != 0 && out && at < hist_cap) {
            out[2 * at] = z;
            out[2 * at + 1] = s_small[z];
        }
        pos += __popc(m);
    }
    // words holding sizes >= 64
    const int64_t w0 = kSmallSizes / 32;
    for (int64_t wc = w0; wc < s.words; wc += 32 * 1024) {
        const int64_t wbase = wc + warp * 1024 + lane;
        uint32_t wd[32];
        int c = 0;
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            const int64_t w = wbase + 32 * k;
            wd[k] = w < s.words ? bw[w] : 0u;
        }
#pragma unroll
        for (int k = 0; k < 32; ++k) c += __popc(wd[k]);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(kAll, c, d);
        __syncthreads();  // the last chunk's s_warp has been read
        if (lane == 0) s_warp[warp] = c;
        __syncthreads();
        int64_t at = pos;
        for (int w = 0; w < 32; ++w) {
            at += w < warp ? s_warp[w] : 0;
            pos += s_warp[w];
        }
        auto place = [&](int64_t w, int bit, int64_t a) {
            const int64_t z = (w << 5) + bit;
            if (out && a < hist_cap) {
                out[2 * a] = z;
                out[2 * a + 1] = cnt[z];
            }
            cnt[z] = 0;
        };
        if (c != 0) {  // the whole warp
#pragma unroll
            for (int k = 0; k < 32; ++k) {
                const uint32_t word = wd[k];
                if (!__any_sync(kAll, word != 0u)) continue;
                const int n = __popc(word);
                int upto = n;  // inclusive prefix over the warp
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int o = __shfl_up_sync(kAll, upto, d);
                    if (lane >= d) upto += o;
                }
                if (word) {
                    const int64_t w = wbase + 32 * k;
                    int64_t a = at + upto - n;
                    bw[w] = 0;
                    const int e = atomicAdd(&s_n, 1);
                    if (e < kWordList) {
                        s_list[e] = make_uint4((unsigned)w, word, (unsigned)a, (unsigned)(a >> 32));
                    } else {
                        for (uint32_t b = word; b; b &= b - 1) place(w, __ffs(b) - 1, a++);
                    }
                }
                at += __shfl_sync(kAll, upto, 31);
            }
        }
        __syncthreads();
        for (int e = warp; e < min(s_n, kWordList); e += 32) {
            const uint4 q = s_list[e];
            if ((q.y >> lane) & 1u) place(q.x, lane, (int64_t)(((uint64_t)q.w << 32) | q.z) + __popc(q.y & below));
        }
        __syncthreads();
        if (threadIdx.x == 0) s_n = 0;
    }
    if (threadIdx.x == 0) {
        if (n_sizes) n_sizes[lat] = pos;
        if (out && pos > hist_cap) atomicExch(err, XY_EINVAL);
    }
}

namespace {

constexpr int64_t kAlign = 256;

int64_t round_up(int64_t b) { return (b + kAlign - 1) / kAlign * kAlign; }

// Edge sites of one tile: a bound on the pieces of the tile that reach its edge.
int64_t edge_sites(int tw, int th) { return (tw <= 2 || th <= 2) ? (int64_t)tw * th : 2 * (int64_t)(tw + th) - 4; }

int64_t list_capacity(int Lx, int Ly, int n_lat)
{
    const int fx = Lx / 32, fy = Ly / 32, rx = Lx % 32, ry = Ly % 32;
    int64_t per = (int64_t)fx * fy * edge_sites(32, 32);
    if (rx) per += (int64_t)fy * edge_sites(rx, 32);
    if (ry) per += (int64_t)fx * edge_sites(32, ry);
    if (rx && ry) per += edge_sites(rx, ry);
    return per * n_lat;
}

}  // namespace

// Copies of the small-size counts per lattice: one per 32 tiles, at most 32.
int small_copies(int Lx, int Ly)
{
    const int64_t tiles = (int64_t)((Lx + 31) / 32) * ((Ly + 31) / 32);
    return (int)std::max<int64_t>(1, std::min<int64_t>(32, tiles / 32));
}

int64_t ccl_scratch_bytes(int Lx, int Ly, int n_lat, int64_t* zeroed_bytes)
{
    const int64_t N = (int64_t)Lx * Ly;
    const int64_t words = (N + 1 + 31) / 32;
    const int64_t z = round_up(4 * (N + 1) * n_lat) + round_up(4 * words * n_lat) +
                      round_up((int64_t)4 * kSmallSizes * small_copies(Lx, Ly) * n_lat);
    if (zeroed_bytes) *zeroed_bytes = z;
    const int64_t cap = list_capacity(Lx, Ly, n_lat);
    const int64_t tiles = (int64_t)((Lx + 31) / 32) * ((Ly + 31) / 32) * n_lat;
    return z + round_up(4 * N * n_lat) + 2 * round_up(8 * cap) + round_up(256 * tiles) + round_up(16 * tiles) + kAlign;
}

CclScratch ccl_scratch_carve(void* base, int Lx, int Ly, int n_lat)
{
    const int64_t N = (int64_t)Lx * Ly;
    CclScratch s{};
    s.words = (N + 1 + 31) / 32;
    s.list_cap = list_capacity(Lx, Ly, n_lat);
    char* p = static_cast<char*>(base);
    s.counts = reinterpret_cast<int32_t*>(p);
    p += round_up(4 * (N + 1) * n_lat);
    s.bits = reinterpret_cast<uint32_t*>(p);
    p += round_up(4 * s.words * n_lat);
    s.copies = small_copies(Lx, Ly);
    s.small = reinterpret_cast<int32_t*>(p);
    p += round_up((int64_t)4 * kSmallSizes * s.copies * n_lat);
    s.entry = reinterpret_cast<int32_t*>(p);
    p += round_up(4 * N * n_lat);
    s.list = reinterpret_cast<int2*>(p);
    p += round_up(8 * s.list_cap);
    s.aux = reinterpret_cast<int2*>(p);
    p += round_up(8 * s.list_cap);
    const int64_t tiles = (int64_t)((Lx + 31) / 32) * ((Ly + 31) / 32) * n_lat;
    s.edge_root = reinterpret_cast<uint16_t*>(p);
    p += round_up(256 * tiles);
    s.edge_spin = reinterpret_cast<uint4*>(p);
    p += round_up(16 * tiles);
    s.list_n = reinterpret_cast<int*>(p);
    return s;
}

cudaError_t launch_ccl(const float* theta, int Lx, int Ly, int n_lat, int32_t* labels, const CclScratch& s,
                       int64_t* hist, int64_t hist_cap, int64_t* n_sizes, int* err, cudaStream_t st)
{
    // every pass runs whether or not sizes are asked for: the size pass also
    // points every merged tile root at its domain's root, which the flattening
    // relies on, and the compaction clears the counts for the next call
    const int64_t N = (int64_t)Lx * Ly;
    const int64_t tiles = (int64_t)((Lx + 31) / 32) * ((Ly + 31) / 32) * n_lat;
    cudaError_t e;
    if ((e = cudaMemsetAsync(s.list_n, 0, sizeof(int), st)) != cudaSuccess) return e;
    ccl_tile_kernel<<<(unsigned)((tiles + kTileWarps - 1) / kTileWarps), 32 * kTileWarps, 0, st>>>(
        theta, Lx, Ly, n_lat, labels, s, err);
    ccl_border_kernel<<<(unsigned)((tiles + 7) / 8), 256, 0, st>>>(Lx, Ly, n_lat, labels, s, hist,
                                                                    hist ? 2 * hist_cap * n_lat : 0, err);
    const unsigned g = (unsigned)std::min<int64_t>((s.list_cap + 255) / 256, 152 * 8);
    ccl_list_size_kernel<<<g, 256, 0, st>>>(N, labels, s, err);
    ccl_list_hist_kernel<<<g, 256, 0, st>>>(N, s, err);
    int shift = 0;
    while ((1 << shift) < Lx) ++shift;
    const auto flatten = (1 << shift) == Lx ? ccl_flatten_kernel<true> : ccl_flatten_kernel<false>;
    flatten<<<(unsigned)((tiles + 7) / 8), 256, 0, st>>>(Lx, Ly, n_lat, 1.0f / (float)Lx, shift, labels);
    ccl_compact_kernel<<<n_lat, 1024, 0, st>>>(N, s, hist, hist_cap, n_sizes, err);
    return cudaGetLastError();
}

}  // namespace xy

// Diagnostics: bound of the union-find loops on the current device
// (iters <= 0 restores the default 2^22).
extern "C" int xy_debug_set_union_limit(int iters)
{
    const int v = iters > 0 ? iters : xy::kMaxUnionIters;
    const cudaError_t e = cudaMemcpyToSymbol(xy::g_union_limit, &v, sizeof(int));
    if (e != cudaSuccess) {
        cudaGetLastError();
        return xy::report_error(XY_ECUDA, cudaGetErrorString(e));
    }
    return XY_OK;
}
