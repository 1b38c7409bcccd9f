// clusters.cu -- cluster-size histogram of one lipid species (section "Cluster
// Analysis methods": clusters of like lipids over the six nearest neighbours, an
// O(n) labelling, the distribution of cluster sizes).
//
// Only the sizes are wanted, so no label of a site ever reaches memory.  The lattice is
// cut into tiles of 32 rows by 8 words (256 sites).  A CTA holds a tile's bits in
// shared memory and unites its runs -- the maximal sequences of the species within a
// 32-site word, found by bit operations -- by a concurrent union-find there: two runs
// of adjacent rows are united once, at the first place where they touch.  A component
// that does not reach its tile's border is complete and goes into the histogram; the
// others become nodes of a small union-find in device memory, which a second kernel
// joins across the borders, a third sums up and a fourth counts.  Trees are joined
// lock-free, the larger root under the smaller by compare-and-swap (as in Jaiganesh &
// Burtscher, ECL-CC, 2018); sizes do not depend on the order.
//
// Bound: the latency of the shared-memory trees; the bits are read twice and a tile
// of 8192 sites leaves about 200 nodes.  8192^2 at 50/50, demixing (GB300, per
// species): 0.51 ms (tiles 0.36, borders, sums and counts about 0.06 each with cold
// caches); 21 ms with one parent entry per site in device memory (the sum over sites 13
// ms, one atomic per site on the largest cluster's root; the unions 5.6; the compaction's
// scan of every size 3.3).  400^2, 40% A: 50 us, 140 before.  Lattices that one CTA's
// shared memory holds are done by one launch: 64^2 11 us, 116 before (five launches, one
// site per thread on 4 CTAs).
#include "klmc_internal.h"

namespace klmc {
namespace {

constexpr int kTileRows = 32, kTileWords = 8;
constexpr int kTileThreads = kTileRows * kTileWords;         // one per word
// Places of a word's sites in the trees: 33, so that one place of all the words of a warp
// lies in 32 banks.  (With 32, all of a column lay in one: columns of single sites, 256 x
// 128, 173 -> 117 us; disordered lattices the same.)
constexpr int kPlaces = 33;
constexpr int kTilePlaces = kPlaces * kTileThreads;
constexpr int kSmallSizes = 256;                             // sizes counted in shared memory first
constexpr int kSmallMaxThreads = 1024;  // words of a lattice that one CTA holds
constexpr int kCountThreads = 512;
constexpr int kTileSmem = kTilePlaces * (4 + 2);
// per word of a small lattice: places (then a histogram), counts (a pair of places each), bits
constexpr int kSmallWordSmem = kPlaces * 4 + (kPlaces + 1) * 2 + 4;

struct CcJob {
    const void *lat;
    int packing, pitch, Lx, Ly, W, species, geometry, helical;
    int tcols, trows, slots;  // tiles across and down; border nodes a tile may have
};

// Word w of row y, a bit per site of the species.
__device__ __forceinline__ uint32_t species_word(const CcJob &J, int y, int w)
{
    const int n = min(32, J.Lx - 32 * w);
    uint32_t v = 0u;
    if (J.packing == kPackBit) {
        v = ((const uint32_t *)J.lat)[(size_t)y * J.pitch + w];
    } else {
        const uint8_t *row = (const uint8_t *)J.lat + (size_t)y * J.pitch + 32 * w;
        if (n == 32 && ((uintptr_t)row & 3u) == 0u) {
            for (int q = 0; q < 8; ++q) {  // four bytes at a time, nonzero bytes to bits
                const uint32_t b = ((const uint32_t *)row)[q];
                const uint32_t t = (((b & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | b) & 0x80808080u;
                v |= ((t >> 7 & 1u) | (t >> 14 & 2u) | (t >> 21 & 4u) | (t >> 28 & 8u)) << (4 * q);
            }
        } else {
            for (int b = 0; b < n; ++b) v |= (row[b] ? 1u : 0u) << b;
        }
    }
    if (J.species == 0) v = ~v;
    return n < 32 ? v & ((1u << n) - 1u) : v;
}

// First site of the run of v that holds bit p.
__device__ __forceinline__ int run_start(uint32_t v, int p)
{
    int z;
    asm("bfind.u32 %0, %1;" : "=r"(z) : "r"(~v & ((1u << p) - 1u)));
    return z + 1;
}

__device__ __forceinline__ int run_length(uint32_t v, int p)
{
    const uint32_t rest = ~(v >> p);
    return rest == 0u ? 32 : __ffs(rest) - 1;
}

// Root of x, shortening the path on the way: every visited node is re-pointed to
// its grandparent (pointer jumping).  That write is always an ancestor, and only
// non-roots are written, so it is safe next to the compare-and-swap on roots.
__device__ __forceinline__ int find_root(volatile int32_t *parent, int x)
{
    int p = parent[x];
    if (p == x) return x;
    int prev = x;
    int next;
    while (p != (next = parent[p])) {
        parent[prev] = next;
        prev = p;
        p = next;
    }
    return p;
}

__device__ __forceinline__ void unite(int32_t *parent, int a, int b)
{
    while (true) {
        a = find_root((volatile int32_t *)parent, a);
        b = find_root((volatile int32_t *)parent, b);
        if (a == b) return;
        if (a < b) {
            const int t = a;
            a = b;
            b = t;
        }
        // a > b: hook root a under b; if a stopped being a root, retry from there.
        const int old = atomicCAS(parent + a, a, b);
        if (old == a) return;
        a = old;
    }
}

// Places where a word v of one row and the word b below it need a union: v's and b's
// runs touch at x (first place of a contact; the rest of it joins the same runs).
__device__ __forceinline__ uint32_t straight_contacts(uint32_t v, uint32_t b)
{
    const uint32_t m = v & b;
    return m & ~(m << 1);
}

// ... and at (x, y), (x-1, y+1) only: bl is b's row moved right by one (its site x-1 at
// x), vl v's.  A straight contact at x (b at x) or at x-1 (v at x-1) joins the same runs.
__device__ __forceinline__ uint32_t slanted_contacts(uint32_t v, uint32_t b, uint32_t vl, uint32_t bl)
{
    return v & bl & ~b & ~vl;
}

// The occupied-size bitmaps: l0 a bit per size, l1 a bit per word of l0, l2 per word of l1.
__device__ __forceinline__ void count_size(const ClusterScratch &s, int size, int n)
{
    if (atomicAdd(s.hist + size, n) != 0) return;
    if (atomicOr(s.l0 + (size >> 5), 1u << (size & 31)) != 0u) return;
    if (atomicOr(s.l1 + (size >> 10), 1u << ((size >> 5) & 31)) != 0u) return;
    atomicOr(s.l2 + (size >> 15), 1u << ((size >> 10) & 31));
}

// Adds len to the 16-bit count of a root, with the border mark in its top bit.
__device__ __forceinline__ void add_count(uint32_t *cnt, int root, uint32_t len, bool border)
{
    const int sh = 16 * (root & 1);
    atomicAdd(cnt + (root >> 1), len << sh);
    if (border) atomicOr(cnt + (root >> 1), 0x8000u << sh);
}

__device__ __forceinline__ uint32_t get_count(const uint32_t *cnt, int i) { return (cnt[i >> 1] >> (16 * (i & 1))) & 0xFFFFu; }

// Border labels of a tile: node of the run that starts at a site of its first and of
// its last row, and of the site in its first and its last column.
struct TileLabels {
    int32_t *top, *bottom, *left, *right;
};

__device__ __forceinline__ TileLabels tile_labels(const CcJob &J, const ClusterScratch &s, int tile)
{
    int32_t *const p = s.labels + (size_t)tile * J.slots;
    const int tw = min(J.Lx, 32 * kTileWords), th = min(J.Ly, kTileRows);
    return {p, p + tw, p + 2 * tw, p + 2 * tw + th};
}

__global__ void __launch_bounds__(kTileThreads, 4)
cc_tiles_kernel(const CcJob J, const ClusterScratch s, int tiles)
{
    extern __shared__ __align__(16) int32_t parent[];  // the places, then the counts
    uint32_t *const cnt = (uint32_t *)(parent + kTilePlaces);
    __shared__ uint32_t bits[kTileRows + 1][kTileWords + 2];  // row and word + 1; zeros around
    __shared__ int small[kSmallSizes];
    __shared__ int nodes;
    const int tid = threadIdx.x;
    const int r = tid / kTileWords, w = tid % kTileWords;
    for (int i = tid; i < kSmallSizes; i += kTileThreads) small[i] = 0;
    for (int i = tid; i < (kTileRows + 1) * (kTileWords + 2); i += kTileThreads) (&bits[0][0])[i] = 0u;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int tr = tile / J.tcols, tc = tile - tr * J.tcols;
        const int y = tr * kTileRows + r, gw = tc * kTileWords + w;
        const int th = min(kTileRows, J.Ly - tr * kTileRows), tw = min(kTileWords, J.W - tc * kTileWords);
        const bool in = r < th && w < tw;
        __syncthreads();
        const uint32_t v = in ? species_word(J, y, gw) : 0u;
        bits[r][w + 1] = v;
        if (tid == 0) nodes = 0;
        const int base = kPlaces * tid;
        for (int k = 4 * tid; k < kTilePlaces; k += 4 * kTileThreads) {  // every site its own root, nothing counted
            *(int4 *)(parent + k) = make_int4(k, k + 1, k + 2, k + 3);
            if (k < kTilePlaces / 2) *(int4 *)(cnt + k) = make_int4(0, 0, 0, 0);
        }
        __syncthreads();
        {
            const uint32_t right = bits[r][w + 2], vleft = bits[r][w], b = bits[r + 1][w + 1], bleft = bits[r + 1][w];
            if ((v >> 31) & right & 1u) unite(parent, base + run_start(v, 31), base + kPlaces);
            const int below = base + kPlaces * kTileWords;
            for (uint32_t m = straight_contacts(v, b); m != 0u; m &= m - 1u) {
                const int p = __ffs(m) - 1;
                unite(parent, base + run_start(v, p), below + run_start(b, p));
            }
            if (J.geometry == kTRI6) {
                for (uint32_t m = slanted_contacts(v, b, (v << 1) | (vleft >> 31), (b << 1) | (bleft >> 31)); m != 0u;
                     m &= m - 1u) {
                    const int p = __ffs(m) - 1;
                    unite(parent, base + run_start(v, p),
                          p > 0 ? below + run_start(b, p - 1) : below - kPlaces + run_start(bleft, 31));
                }
            }
        }
        __syncthreads();
        // A run's sites go to its root; runs on the border mark it.
        const int last = min(32, J.Lx - 32 * gw) - 1;  // the word's last column
        const uint32_t starts = v & ~(v << 1);
        for (uint32_t m = starts; m != 0u; m &= m - 1u) {
            const int p = __ffs(m) - 1, len = run_length(v, p);
            const bool border = r == 0 || r == th - 1 || (w == 0 && p == 0) || (w == tw - 1 && p + len - 1 == last);
            const int root = find_root((volatile int32_t *)parent, base + p);
            add_count(cnt, root, (uint32_t)len, border);
        }
        __syncthreads();
        const size_t node0 = (size_t)tile * J.slots;
        for (uint32_t m = starts; m != 0u; m &= m - 1u) {
            const int i = base + __ffs(m) - 1;
            if (parent[i] != i) continue;
            const uint32_t c = get_count(cnt, i);
            const int size = (int)(c & 0x7FFFu);
            if (c & 0x8000u) {
                const int k = atomicAdd(&nodes, 1);
                s.parent[node0 + k] = (int32_t)(node0 + k);
                s.csize[node0 + k] = size;
                // the root's count becomes its node (no other thread reads it before the barrier)
                const int sh = 16 * (i & 1);
                atomicAdd(cnt + (i >> 1), (uint32_t)k << sh);
                atomicSub(cnt + (i >> 1), c << sh);
            } else if (size < kSmallSizes) {
                atomicAdd(&small[size], 1);
            } else {
                count_size(s, size, 1);
            }
        }
        __syncthreads();
        if (tid == 0) s.nodes[tile] = nodes;
        const TileLabels L = tile_labels(J, s, tile);
        auto node_of = [&](int i) { return (int32_t)(node0 + get_count(cnt, find_root((volatile int32_t *)parent, i))); };
        if (in && (r == 0 || r == th - 1)) {
            for (uint32_t m = starts; m != 0u; m &= m - 1u) {
                const int p = __ffs(m) - 1;
                const int32_t id = node_of(base + p);
                if (r == 0) L.top[32 * w + p] = id;
                if (r == th - 1) L.bottom[32 * w + p] = id;
            }
        }
        if (in && w == 0 && (v & 1u)) L.left[r] = node_of(base);
        if (in && w == tw - 1 && ((v >> last) & 1u)) L.right[r] = node_of(base + run_start(v, last));
    }
    __syncthreads();
    for (int i = tid; i < kSmallSizes; i += kTileThreads)
        if (small[i] != 0) count_size(s, i, small[i]);
}

// Unions across tile borders.  Items 0 .. kParts trows W - 1: a part of a word of a tile
// row's last row against the row below it (a union is a chain of waits for memory, and an
// ordered lattice has 16 a word; 400^2, columns of single sites, with whole words 186 us,
// in 8 parts 91, in 16 parts 85 but 8192^2 demixed slower); then tcols Ly items: a row at the right end of a tile column
// against the first site of the next.  Around the lattice's sides the x wrap stays in
// its row (periodic) or carries into the next or previous row (helical).
constexpr int kParts = 8;

__global__ void cc_merge_kernel(const CcJob J, const ClusterScratch s, long long items)
{
    const int nlast = J.Lx - 32 * (J.W - 1);
    for (long long it = blockIdx.x * (long long)blockDim.x + threadIdx.x; it < items;
         it += (long long)gridDim.x * blockDim.x) {
        const long long words = (long long)J.trows * J.W;
        if (it < kParts * words) {
            const int tr = (int)(it / kParts / J.W), w = (int)(it / kParts - (long long)tr * J.W);
            const uint32_t part = (0xFFFFFFFFu >> (32 - 32 / kParts)) << (32 / kParts * (int)(it % kParts));
            const int y = min((tr + 1) * kTileRows, J.Ly) - 1, yn = y + 1 == J.Ly ? 0 : y + 1;
            const int trn = tr + 1 == J.trows ? 0 : tr + 1;
            const int tc = w / kTileWords, x0 = 32 * (w - tc * kTileWords);
            const uint32_t v = species_word(J, y, w), b = species_word(J, yn, w);
            const TileLabels A = tile_labels(J, s, tr * J.tcols + tc), B = tile_labels(J, s, trn * J.tcols + tc);
            for (uint32_t m = straight_contacts(v, b) & part; m != 0u; m &= m - 1u) {
                const int p = __ffs(m) - 1;
                unite(s.parent, A.bottom[x0 + run_start(v, p)], B.top[x0 + run_start(b, p)]);
            }
            if (J.geometry != kTRI6) continue;
            // the last site of the word to the left (none at x = 0 of a helical lattice)
            const int wl = w == 0 ? J.W - 1 : w - 1, end = w == 0 ? nlast - 1 : 31;
            const bool left = w > 0 || !J.helical;
            const uint32_t vl = left ? (species_word(J, y, wl) >> end) & 1u : 0u;
            const uint32_t bw = left ? species_word(J, yn, wl) : 0u;
            for (uint32_t m = slanted_contacts(v, b, (v << 1) | vl, (b << 1) | ((bw >> end) & 1u)) & part; m != 0u;
                 m &= m - 1u) {
                const int p = __ffs(m) - 1;
                int32_t other;
                if (p > 0) {
                    other = B.top[x0 + run_start(b, p - 1)];
                } else {
                    const int tl = wl / kTileWords;
                    other = tile_labels(J, s, trn * J.tcols + tl).top[32 * (wl - tl * kTileWords) + run_start(bw, end)];
                }
                unite(s.parent, A.bottom[x0 + run_start(v, p)], other);
            }
        } else {
            const long long k = it - kParts * words;
            const int tc = (int)(k / J.Ly), y = (int)(k - (long long)tc * J.Ly);
            const bool wrap = tc + 1 == J.tcols;
            const int tcn = wrap ? 0 : tc + 1;
            const int w = wrap ? J.W - 1 : (tc + 1) * kTileWords - 1, end = wrap ? nlast - 1 : 31;
            const int wn = tcn * kTileWords;
            const int tr = y / kTileRows, r = y - tr * kTileRows;
            const int yn = y + 1 == J.Ly ? 0 : y + 1;
            const int trn = yn / kTileRows, rn = yn - trn * kTileRows;
            const bool here = (species_word(J, y, w) >> end) & 1u;  // the column's last site in row y
            const bool next = species_word(J, y, wn) & 1u;            // the next column's first site in row y
            const int32_t *const right = tile_labels(J, s, tr * J.tcols + tc).right;
            if (wrap && J.helical) {
                // (Lx-1, y): its right neighbour is (0, y+1), its (1,-1) neighbour (0, y)
                if (here && (species_word(J, yn, wn) & 1u))
                    unite(s.parent, right[r], tile_labels(J, s, trn * J.tcols + tcn).left[rn]);
                if (here && next && J.geometry == kTRI6)
                    unite(s.parent, right[r], tile_labels(J, s, tr * J.tcols + tcn).left[r]);
                continue;
            }
            if (!next) continue;
            const int32_t id = tile_labels(J, s, tr * J.tcols + tcn).left[r];
            if (here) unite(s.parent, right[r], id);
            // (x, y) and (x-1, y+1) of the column before, inside a tile row
            if (J.geometry == kTRI6 && y + 1 < J.Ly && trn == tr && ((species_word(J, yn, w) >> end) & 1u))
                unite(s.parent, right[r + 1], id);
        }
    }
}

// Sizes of the nodes go to their roots.  Most nodes of a warp belong to one large
// cluster: the warp adds up those that share its first root.
__global__ void cc_sum_kernel(const ClusterScratch s, int tiles, int slots)
{
    const int lane = threadIdx.x & 31;
    const int warps = (int)(gridDim.x * blockDim.x) >> 5;
    for (int tile = (int)(blockIdx.x * blockDim.x + threadIdx.x) >> 5; tile < tiles; tile += warps) {
        const int n = s.nodes[tile];
        const size_t node0 = (size_t)tile * slots;
        for (int k0 = 0; k0 < n; k0 += 32) {
            const int k = k0 + lane;
            int root = -1, size = 0;
            if (k < n) {
                const int id = (int)(node0 + k);
                root = find_root((volatile int32_t *)s.parent, id);
                if (root == id) root = -1;  // its own size is there already
                else size = s.csize[id];
            }
            const unsigned has = __ballot_sync(0xFFFFFFFFu, root >= 0);
            if (has == 0u) continue;
            const int first = __shfl_sync(0xFFFFFFFFu, root, __ffs(has) - 1);
            int sum = root == first ? size : 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
            if (lane == 0) atomicAdd(s.csize + first, sum);
            if (root >= 0 && root != first) atomicAdd(s.csize + root, size);
        }
    }
}

// Ascending (size, count) pairs from the occupied-size bitmaps, by one CTA of
// kCountThreads; clears what it reads.  A word of l2 covers a chunk of 1024 words of
// l0; empty chunks are skipped.  In a chunk every warp takes words of l0, a lane per size.
__device__ void compact(const ClusterScratch &s, long long *sizes, long long *counts, long long capacity,
                        long long *n_distinct)
{
    constexpr int kWarps = kCountThreads / 32, kPer = 1024 / kCountThreads;
    __shared__ uint32_t words[1024];
    __shared__ int offset[1024];
    __shared__ int warp_tot[kWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long chunks = (s.n_species_max >> 15) + 1;
    long long base = 0;
    for (long long c0 = 0; c0 < chunks; c0 += kCountThreads) {
        const bool full = c0 + tid < chunks && __ldcg(s.l2 + c0 + tid) != 0u;
        __shared__ uint32_t todo[kWarps];
        const unsigned any = __ballot_sync(0xFFFFFFFFu, full);
        __syncthreads();
        if (lane == 0) todo[warp] = any;
        __syncthreads();
        for (int g = 0; g < kWarps; ++g) {
            for (uint32_t m = todo[g]; m != 0u; m &= m - 1u) {
                const long long chunk = c0 + 32 * g + __ffs(m) - 1;
                const long long nwords = (s.n_species_max >> 5) + 1;
                uint32_t v[kPer];
                int sum = 0;
#pragma unroll
                for (int q = 0; q < kPer; ++q) {  // words kPer tid .. of the chunk
                    const long long w = chunk * 1024 + kPer * tid + q;
                    v[q] = w < nwords ? __ldcg(s.l0 + w) : 0u;
                    sum += __popc(v[q]);
                }
                int incl = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                    if (lane >= o) incl += t;
                }
                if (lane == 31) warp_tot[warp] = incl;
                __syncthreads();
                int before = incl - sum, total = 0;
                for (int k = 0; k < kWarps; ++k) {
                    if (k < warp) before += warp_tot[k];
                    total += warp_tot[k];
                }
#pragma unroll
                for (int q = 0; q < kPer; ++q) {
                    words[kPer * tid + q] = v[q];
                    offset[kPer * tid + q] = before;
                    before += __popc(v[q]);
                }
                __syncthreads();
                for (int i = warp; i < 1024; i += kWarps) {
                    const uint32_t bitsw = words[i];
                    if (bitsw == 0u) continue;
                    const long long w = chunk * 1024 + i;
                    if ((bitsw >> lane) & 1u) {
                        const long long size = 32 * w + lane;
                        const long long pos = base + offset[i] + __popc(bitsw & ((1u << lane) - 1u));
                        const int n = __ldcg(s.hist + size);
                        s.hist[size] = 0;
                        if (pos < capacity) {
                            sizes[pos] = size;
                            counts[pos] = n;
                        }
                    }
                    if (lane == 0) s.l0[w] = 0u;
                }
                for (int i = tid; i < 32; i += kCountThreads)
                    if (chunk * 32 + i <= (s.n_species_max >> 10)) s.l1[chunk * 32 + i] = 0u;
                if (tid == 0) s.l2[chunk] = 0u;
                base += total;
                __syncthreads();
            }
        }
    }
    if (tid == 0) *n_distinct = base;
}

// Counts the roots' sizes; the last CTA to finish writes the sparse histogram.
__global__ void __launch_bounds__(kCountThreads)
cc_count_kernel(const ClusterScratch s, int tiles, int slots, long long *sizes, long long *counts, long long capacity,
                long long *n_distinct)
{
    __shared__ int small[kSmallSizes];
    __shared__ bool last;
    for (int i = threadIdx.x; i < kSmallSizes; i += kCountThreads) small[i] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int warps = (int)(gridDim.x * kCountThreads) >> 5;
    for (int tile = (int)(blockIdx.x * kCountThreads + threadIdx.x) >> 5; tile < tiles; tile += warps) {
        const int n = s.nodes[tile];
        const size_t node0 = (size_t)tile * slots;
        for (int k = lane; k < n; k += 32) {
            const int id = (int)(node0 + k);
            if (s.parent[id] != id) continue;
            const int size = s.csize[id];
            if (size < kSmallSizes) atomicAdd(&small[size], 1);
            else count_size(s, size, 1);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kSmallSizes; i += kCountThreads)
        if (small[i] != 0) count_size(s, i, small[i]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(s.done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    compact(s, sizes, counts, capacity, n_distinct);
    if (threadIdx.x == 0) *s.done = 0u;
}

// A lattice of at most 8 words by 1024 words in all, in one CTA: unions (with the
// wraps), sizes, a histogram in the trees' memory and its compaction.  `parts` threads
// (a power of two, at most 4) share a word, each with the contacts and the runs' starts in
// its part: a word's unions wait for each other.  (64^2 with one / 4 / 8 threads: demixed
// 19 / 12 / 12 us, columns of single sites 82 / 25 / 13, rows 6.7 / 6.5 / 8.5.)
__global__ void __launch_bounds__(kSmallMaxThreads, 1)
cc_small_kernel(const CcJob J, int parts, long long *sizes, long long *counts, long long capacity, long long *n_distinct)
{
    extern __shared__ __align__(16) int32_t parent[];  // the words' places, then the counts
    const int words = J.W * J.Ly, places = kPlaces * words;  // entry e of the histogram is at e + e / 32
    uint32_t *const cnt = (uint32_t *)(parent + places);
    uint32_t *const bits = cnt + (places + 1) / 2;
    __shared__ int warp_tot[32];
    const int tid = threadIdx.x, T = blockDim.x;
    const int word = tid / parts, y = word / J.W, w = word - y * J.W;
    const bool in = word < words;
    const uint32_t v = in ? species_word(J, y, w) : 0u;
    const int part0 = 32 / parts * (tid & (parts - 1));  // its first bit
    const uint32_t part = (0xFFFFFFFFu >> (32 - 32 / parts)) << part0;
    if (in && part0 == 0) bits[word] = v;
    for (int i = tid; i < places; i += T) parent[i] = i;
    for (int i = tid; i < (places + 1) / 2; i += T) cnt[i] = 0u;
    __syncthreads();
    if (in) {
        const int nlast = J.Lx - 32 * (J.W - 1);
        const int yn = y + 1 == J.Ly ? 0 : y + 1;
        const bool first = w == 0, lastw = w == J.W - 1;
        const int end = lastw ? nlast - 1 : 31;  // the word's last site
        const int base = kPlaces * word, below = kPlaces * (yn * J.W + w);
        const uint32_t b = bits[yn * J.W + w];
        const int lw = first ? J.W - 1 : w - 1, lend = first ? nlast - 1 : 31;
        // the site to the right of the word's last one
        const int rw = lastw ? 0 : w + 1, ry = lastw && J.helical ? yn : y;
        if (((v & part) >> end & 1u) && (bits[ry * J.W + rw] & 1u))
            unite(parent, base + run_start(v, end), kPlaces * (ry * J.W + rw));
        for (uint32_t m = straight_contacts(v, b) & part; m != 0u; m &= m - 1u) {
            const int p = __ffs(m) - 1;
            unite(parent, base + run_start(v, p), below + run_start(b, p));
        }
        if (J.geometry == kTRI6) {
            // (x, y) and (x-1, y+1); at x = 0 of a helical lattice that is (Lx-1, y)
            const int sy = first && J.helical ? y : yn;
            const uint32_t sl = bits[sy * J.W + lw], vl = bits[y * J.W + lw];
            const bool carry = first && J.helical;
            const uint32_t bl = (b << 1) | ((sl >> lend) & 1u);
            uint32_t m = slanted_contacts(v, b, (v << 1) | ((vl >> lend) & 1u), bl);
            if (carry) m = (m & ~1u) | (v & bl & 1u);  // its own bond: no straight contact stands for it
            for (m &= part; m != 0u; m &= m - 1u) {
                const int p = __ffs(m) - 1;
                unite(parent, base + run_start(v, p),
                      p > 0 ? below + run_start(b, p - 1) : kPlaces * (sy * J.W + lw) + run_start(sl, lend));
            }
        }
    }
    __syncthreads();
    const uint32_t starts = v & ~(v << 1) & part;
    for (uint32_t m = starts; m != 0u; m &= m - 1u) {
        const int p = __ffs(m) - 1;
        add_count(cnt, find_root((volatile int32_t *)parent, kPlaces * word + p), (uint32_t)run_length(v, p), false);
    }
    __syncthreads();
    for (int i = tid; i < places; i += T) parent[i] = 0;  // now the histogram: entry size - 1
    __syncthreads();
    for (uint32_t m = starts; m != 0u; m &= m - 1u) {
        const uint32_t c = get_count(cnt, kPlaces * word + __ffs(m) - 1);  // nonzero at roots only
        if (c != 0u) atomicAdd(parent + (c - 1) + ((c - 1) >> 5), 1);
    }
    __syncthreads();
    // Compaction: every thread the entries of one contiguous part.
    const int lane = tid & 31, warp = tid >> 5, nw = T >> 5;
    const int sites = 32 * words, per = (sites + T - 1) / T, e0 = min(tid * per, sites), e1 = min(e0 + per, sites);
    int n = 0;
    for (int e = e0; e < e1; ++e) n += parent[e + (e >> 5)] != 0;
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    long long pos = incl - n;
    int total = 0;
    for (int k = 0; k < nw; ++k) {
        if (k < warp) pos += warp_tot[k];
        total += warp_tot[k];
    }
    for (int e = e0; e < e1; ++e) {
        const int c = parent[e + (e >> 5)];
        if (c == 0) continue;
        if (pos < capacity) {
            sizes[pos] = e + 1;
            counts[pos] = c;
        }
        ++pos;
    }
    if (tid == 0) *n_distinct = total;
}

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

// Border nodes and tiles of any lattice of N sites: a tile of tw x th sites has
// 2 (tw + th) border sites; strips of 4 sites and small lattices have the most for their size.
long long max_nodes(long long N) { return (3 * N + 4) / 5 + 2048; }
long long max_tiles(long long N) { return N / 96 + 64; }

}  // namespace

size_t cluster_scratch_bytes(long long N, long long n_species_max)
{
    ClusterScratch s;
    cluster_scratch_carve(nullptr, N, n_species_max, &s);
    return (size_t)(uintptr_t)s.end;
}

void cluster_scratch_carve(void *base, long long N, long long n_species_max, ClusterScratch *s)
{
    char *p = (char *)base;
    auto take = [&](size_t bytes) {
        char *const q = p;
        p += align256(bytes);
        return q;
    };
    s->n_species_max = n_species_max;
    s->hist = (int32_t *)take((size_t)(n_species_max + 1) * 4);
    s->l0 = (uint32_t *)take((size_t)((n_species_max >> 5) + 1) * 4);
    s->l1 = (uint32_t *)take((size_t)((n_species_max >> 10) + 1) * 4);
    s->l2 = (uint32_t *)take((size_t)((n_species_max >> 15) + 1) * 4);
    s->done = (uint32_t *)take(4);
    s->zero_end = p;
    s->parent = (int32_t *)take((size_t)max_nodes(N) * 4);
    s->csize = (int32_t *)take((size_t)max_nodes(N) * 4);
    s->labels = (int32_t *)take((size_t)max_nodes(N) * 4);
    s->nodes = (int32_t *)take((size_t)max_tiles(N) * 4);
    s->end = p;
}

cudaError_t cluster_scratch_clear(const ClusterScratch &s, cudaStream_t stream)
{
    return cudaMemsetAsync(s.hist, 0, (size_t)((char *)s.zero_end - (char *)s.hist), stream);
}

cudaError_t launch_cluster_histogram(const void *lat, int packing, int Lx, int Ly, int pitch,
                                     int geometry, int species, const ClusterScratch &s,
                                     long long *sizes, long long *counts, long long capacity,
                                     long long *n_distinct, cudaStream_t stream, int helical)
{
    const int W = (Lx + 31) / 32;
    CcJob J = {lat, packing, pitch, Lx, Ly, W, species, geometry, helical, 0, 0, 0};
    static thread_local int configured_device = -1;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess && configured_device != dev) {
        e = cudaFuncSetAttribute(cc_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kSmallMaxThreads * kSmallWordSmem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(cc_tiles_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTileSmem);
        if (e == cudaSuccess) configured_device = dev;
    }
    if (e != cudaSuccess) return e;
    if (W <= kTileWords && (long long)W * Ly <= kSmallMaxThreads) {
        int parts = 1;
        while (parts < 4 && 2 * parts * W * Ly <= kSmallMaxThreads) parts *= 2;
        const int words = W * Ly, threads = (parts * words + 31) / 32 * 32;
        cc_small_kernel<<<1, threads, (size_t)words * kSmallWordSmem, stream>>>(J, parts, sizes, counts,
                                                                                capacity, n_distinct);
        return cudaGetLastError();
    }
    J.tcols = (W + kTileWords - 1) / kTileWords;
    J.trows = (Ly + kTileRows - 1) / kTileRows;
    J.slots = 2 * ((Lx < 32 * kTileWords ? Lx : 32 * kTileWords) + (Ly < kTileRows ? Ly : kTileRows));
    const int tiles = J.tcols * J.trows;
    auto grid = [](long long n, long long most) { return (int)(n < 1 ? 1 : (n < most ? n : most)); };
    cc_tiles_kernel<<<grid(tiles, 152 * 4), kTileThreads, kTileSmem, stream>>>(J, s, tiles);
    const long long items = (long long)kParts * J.trows * W + (long long)J.tcols * Ly;
    cc_merge_kernel<<<grid((items + 127) / 128, 152 * 16), 128, 0, stream>>>(J, s, items);
    cc_sum_kernel<<<grid((tiles + 3) / 4, 152 * 16), 128, 0, stream>>>(s, tiles, J.slots);
    cc_count_kernel<<<grid((tiles + 15) / 16, 152 * 2), kCountThreads, 0, stream>>>(s, tiles, J.slots, sizes, counts,
                                                                                  capacity, n_distinct);
    return cudaGetLastError();
}

}  // namespace klmc
