// lattice_ops.cu -- initial placement, energy recount, and lattice (un)packing.
//
// Initial placement (Fig. 2: lipids randomly distributed over the lattice, the
// number of each type fixed): every site i gets the 96-bit key (K64_i, i), K64_i a
// 64-bit Philox value; the n_A sites with the smallest keys are A.  The keys are
// distinct, so this is a uniformly random n_A-subset.  It is computed by a radix
// select over digits of 12 bits (8 for small lattices), most significant first,
// recomputing the keys in every pass instead of storing them; it stops as soon as the
// selected bucket is taken whole.  The last CTA of a pass picks its digit, and that of
// the last launched pass finishes alone in the rare case that is left: two launches
// per pass for all 96 bits took 90 of the 270 us of a new 1000^2 lattice.
#include <string.h>

#include "klmc_internal.h"
#include "philox.cuh"

namespace klmc {
namespace {

constexpr int kBlock = 256;


// Placement key of site i: Philox counter {i, 0xFFFFFFFF, 0, 0}, words w1:w0.
__device__ __forceinline__ unsigned long long site_key(uint32_t i, uint32_t k0, uint32_t k1)
{
    const Philox4 w = philox4(i, 0xFFFFFFFFu, 0u, 0u, k0, k1);
    return ((unsigned long long)w.v[1] << 32) | w.v[0];
}

struct SelectState {
    unsigned long long p_hi;  // fixed key bits, left-aligned in the 96-bit key
    unsigned int p_lo;
    int nbits;                // number of fixed bits
    long long k;              // rank (1-based) still to reach inside the prefix bucket
    int done;
    unsigned int finished;    // CTAs of the running pass that have added their counts
    unsigned int hist[256];   // counts of an 8-bit pass, zero between passes
};

__device__ __forceinline__ void key_masks(int nbits, unsigned long long &mh, unsigned int &ml)
{
    mh = nbits >= 64 ? ~0ull : (nbits == 0 ? 0ull : (~0ull << (64 - nbits)));
    ml = nbits <= 64 ? 0u : (nbits >= 96 ? ~0u : (~0u << (96 - nbits)));
}

// Adds the digits [nbits, nbits + BITS) of the keys of sites first, first + step, ..
// that share the prefix to the counts h.
template <int BITS>
__device__ __forceinline__ void count_digits(unsigned int *h, long long N, long long first, long long step, uint32_t k0,
                                             uint32_t k1, const SelectState &st)
{
    unsigned long long mh;
    unsigned int ml;
    key_masks(st.nbits, mh, ml);
    const int sh = max(96 - BITS - st.nbits, 0);  // the digit's place in the 96-bit key
    for (long long i = first; i < N; i += step) {
        const unsigned long long kh = site_key((uint32_t)i, k0, k1);
        const unsigned int kl = (unsigned int)i;
        if ((kh & mh) != st.p_hi || (kl & ml) != st.p_lo) continue;
        const unsigned long long at = sh >= 32 ? kh >> (sh - 32) : ((kh << 32) | kl) >> sh;
        atomicAdd(&h[(unsigned int)at & ((1u << BITS) - 1u)], 1u);
    }
}

template <int BITS>
__global__ void __launch_bounds__(kBlock)
select_kernel(long long N, uint32_t k0, uint32_t k1, SelectState *st, unsigned int *hist, int finish)
{
    constexpr int kDigits = 1 << BITS, kPer = kDigits / kBlock;
    __shared__ unsigned int h[kDigits];
    __shared__ unsigned int part[kBlock];
    __shared__ SelectState S;  // (its counts unused)
    __shared__ bool last;
    const int tid = threadIdx.x;
    if (st->done) return;
    if (tid == 0) {
        S.p_hi = st->p_hi;
        S.p_lo = st->p_lo;
        S.nbits = st->nbits;
        S.k = st->k;
        S.done = 0;
    }
    for (int b = tid; b < kDigits; b += kBlock) h[b] = 0u;
    __syncthreads();
    count_digits<BITS>(h, N, blockIdx.x * (long long)kBlock + tid, (long long)gridDim.x * kBlock, k0, k1, S);
    __syncthreads();
    for (int b = tid; b < kDigits; b += kBlock)
        if (h[b]) atomicAdd(&hist[b], h[b]);
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(&st->finished, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int b = tid; b < kDigits; b += kBlock) {
        h[b] = __ldcg(&hist[b]);
        hist[b] = 0u;
    }
    while (true) {
        __syncthreads();
        // The digit whose bucket holds the rank: every thread sums kPer counts.
        unsigned int c[kPer], sum = 0u;
#pragma unroll
        for (int q = 0; q < kPer; ++q) sum += c[q] = h[kPer * tid + q];
        part[tid] = sum;
        __syncthreads();
        for (int o = 1; o < kBlock; o <<= 1) {  // inclusive scan
            const unsigned int add = tid >= o ? part[tid - o] : 0u;
            __syncthreads();
            part[tid] += add;
            __syncthreads();
        }
        const long long k = S.k, upto = (long long)part[tid];
        const int nbits = S.nbits;
        long long before = upto - sum;
        __syncthreads();  // every thread has the rank
        if (before < k && k <= upto) {
            unsigned int digit = kPer * tid, n = 0u;
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                n = c[q];
                if (before + n >= k) break;
                before += n;
                ++digit;
            }
            const int sh = max(96 - BITS - nbits, 0);  // (a last digit repeats fixed bits)
            if (sh >= 32) {
                S.p_hi |= (unsigned long long)digit << (sh - 32);
            } else {
                const unsigned long long low = (unsigned long long)digit << sh;  // may reach into the high word
                S.p_hi |= low >> 32;
                S.p_lo |= (unsigned int)low;
            }
            S.k = k - before;
            S.nbits = nbits + BITS;
            S.done = (long long)n == k - before || S.nbits >= 96;
        }
        __syncthreads();
        if (S.done || !finish) break;
        for (int b = tid; b < kDigits; b += kBlock) h[b] = 0u;
        __syncthreads();
        count_digits<BITS>(h, N, tid, kBlock, k0, k1, S);
    }
    if (tid == 0) {
        st->p_hi = S.p_hi;
        st->p_lo = S.p_lo;
        st->nbits = S.nbits;
        st->k = S.k;
        st->done = S.done;
        st->finished = 0u;
    }
}

__global__ void select_start_kernel(SelectState *st, long long k)
{
    unsigned int *const words = (unsigned int *)st;
    for (int i = threadIdx.x; i < (int)(sizeof(SelectState) / 4); i += blockDim.x) words[i] = 0u;
    __syncthreads();
    if (threadIdx.x == 0) st->k = k;
}

// mode 0: none are A; 1: all are A; 2: A iff the key's fixed top bits <= prefix.
__device__ __forceinline__ uint32_t is_A(uint32_t i, uint32_t k0, uint32_t k1, int mode,
                                         const SelectState &st)
{
    if (mode != 2) return (uint32_t)mode;
    unsigned long long mh;
    unsigned int ml;
    key_masks(st.nbits, mh, ml);
    const unsigned long long kh = site_key(i, k0, k1) & mh;
    const unsigned int kl = i & ml;
    return (kh < st.p_hi || (kh == st.p_hi && kl <= st.p_lo)) ? 1u : 0u;
}

__global__ void mark_kernel(void *lat, int packing, int Lx, int Ly, int pitch, uint32_t k0,
                            uint32_t k1, int mode, const SelectState *st_ptr)
{
    SelectState st;
    st.p_hi = st_ptr->p_hi;
    st.p_lo = st_ptr->p_lo;
    st.nbits = st_ptr->nbits;
    if (packing == kPackBit) {
        const int W = (Lx + 31) / 32;
        const long long nwords = (long long)W * Ly;
        const int lane = threadIdx.x & 31;
        for (long long wi = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; wi < nwords;
             wi += ((long long)gridDim.x * blockDim.x) >> 5) {
            const int y = (int)(wi / W), w = (int)(wi - (long long)y * W);
            const int x = 32 * w + lane;
            uint32_t a = 0u;
            if (x < Lx) a = is_A((uint32_t)((long long)y * Lx + x), k0, k1, mode, st);
            const uint32_t word = __ballot_sync(0xFFFFFFFFu, a != 0u);
            if (lane == 0) ((uint32_t *)lat)[(size_t)y * pitch + w] = word;
        }
    } else {
        const long long N = (long long)Lx * Ly;
        for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N;
             i += (long long)gridDim.x * blockDim.x) {
            const int y = (int)(i / Lx), x = (int)(i - (long long)y * Lx);
            ((uint8_t *)lat)[(size_t)y * pitch + x] = (uint8_t)is_A((uint32_t)i, k0, k1, mode, st);
        }
    }
}

__device__ __forceinline__ uint32_t site_at(const void *lat, int packing, int pitch, int x, int y)
{
    if (packing == kPackBit) {
        const uint32_t *row = (const uint32_t *)lat + (size_t)y * pitch;
        return (row[x >> 5] >> (x & 31)) & 1u;
    }
    return ((const uint8_t *)lat)[(size_t)y * pitch + x] ? 1u : 0u;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

__device__ __forceinline__ void block_add(long long v, long long *out)
{
    __shared__ long long part[32];
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        long long s = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0;
        s = warp_sum(s);
        if (threadIdx.x == 0 && s != 0) atomicAdd((unsigned long long *)out, (unsigned long long)s);
    }
}

// Bits 0..3: which of the four bytes of b are not zero.
__device__ __forceinline__ uint32_t nonzero_bytes(uint32_t b)
{
    const uint32_t t = ((((b & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | b) >> 7) & 0x01010101u;
    return (t * 0x01020408u) >> 24;  // byte k's bit to bit 24 + k; nothing else lands there
}

// Bits 0..15: which of the sixteen bytes of v are not zero.
__device__ __forceinline__ uint32_t nonzero_bytes(uint4 v)
{
    return nonzero_bytes(v.x) | (nonzero_bytes(v.y) << 4) | (nonzero_bytes(v.z) << 8) | (nonzero_bytes(v.w) << 12);
}

// Four bytes of 0 or 1 from the bits 0..3 of n.
__device__ __forceinline__ uint32_t spread_bits(uint32_t n) { return ((n & 15u) * 0x00204081u) & 0x01010101u; }

// Word w (32 sites) of row y of the store, the bits past the row's end zero.
__device__ __forceinline__ uint32_t site_word(const void *lat, int packing, int pitch, int Lx, int y, int w)
{
    const int n = min(32, Lx - 32 * w);
    uint32_t v = 0u;
    if (packing == kPackBit) {
        v = ((const uint32_t *)lat)[(size_t)y * pitch + w];
    } else {
        const uint8_t *const row = (const uint8_t *)lat + (size_t)y * pitch + 32 * w;
        // rows are padded with zeros to 16 bytes (one or two loads: the energy of a 5000 x 33 byte
        // store in 18 us, with eight loads 25)
        if ((((uintptr_t)row) & 15u) == 0u) {
            const uint4 *const part = (const uint4 *)row;
            v = nonzero_bytes(part[0]);
            if (n > 16) v |= nonzero_bytes(part[1]) << 16;
        } else if ((((uintptr_t)row) & 3u) == 0u) {
            for (int q = 0; 4 * q < n; ++q) v |= nonzero_bytes(((const uint32_t *)row)[q]) << (4 * q);
        } else {
            for (int b = 0; b < n; ++b) v |= (row[b] ? 1u : 0u) << b;
        }
    }
    return n < 32 ? v & ((1u << n) - 1u) : v;
}

// A word's sites and, at each site's place, its neighbours' in the six directions (1,0),
// (-1,0), (0,1), (0,-1), (1,-1), (-1,1); periodic wrap, or the helical wrap of x into
// the next or previous row.
struct WordNeighbours {
    uint32_t v, valid, nb[6];
};

__device__ __forceinline__ WordNeighbours word_neighbours(const void *lat, int packing, int pitch, int Lx, int Ly, int W,
                                                          int helical, int y, int w, bool left)
{
    WordNeighbours N;
    const int n = min(32, Lx - 32 * w);
    N.valid = n == 32 ? 0xFFFFFFFFu : (1u << n) - 1u;
    const int yp = y + 1 == Ly ? 0 : y + 1, ym = y == 0 ? Ly - 1 : y - 1;
    N.v = site_word(lat, packing, pitch, Lx, y, w);
    const uint32_t p = site_word(lat, packing, pitch, Lx, yp, w), m = site_word(lat, packing, pitch, Lx, ym, w);
    const bool lastw = w == W - 1, firstw = w == 0;
    const int xr = lastw ? 0 : 32 * w + 32, xl = firstw ? Lx - 1 : 32 * w - 1;
    const bool cr = lastw && helical, cl = firstw && helical;
    const uint32_t r0 = site_at(lat, packing, pitch, xr, cr ? yp : y), rm = site_at(lat, packing, pitch, xr, cr ? y : ym);
    N.nb[0] = (N.v >> 1) | (r0 << (n - 1));
    N.nb[2] = p;
    N.nb[3] = m;
    N.nb[4] = (m >> 1) | (rm << (n - 1));
    N.nb[1] = N.nb[5] = 0u;
    if (left) {
        N.nb[1] = (N.v << 1) | site_at(lat, packing, pitch, xl, cl ? ym : y);
        N.nb[5] = (p << 1) | site_at(lat, packing, pitch, xl, cl ? y : yp);
    }
    return N;
}

// Unlike bonds {i, i+o}, o in (1,0), (0,1) and, for TRI6, (1,-1), each once, into *unlike,
// and the A sites into *sites_A; either may be null.  A thread per 32-site word: per
// site, with its division and its single-bit loads, 8192^2 took 361 us for the bonds and
// 227 us for the sites; now 16 us for both.
__global__ void tally_kernel(const void *lat, int packing, int Lx, int Ly, int pitch, int geometry, int helical,
                             long long *unlike, long long *sites_A)
{
    const int W = (Lx + 31) / 32;
    const long long nwords = (long long)W * Ly;
    long long n = 0, nA = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nwords;
         i += (long long)gridDim.x * blockDim.x) {
        const int y = (int)((uint32_t)i / (uint32_t)W), w = (int)((uint32_t)i - (uint32_t)y * (uint32_t)W);
        if (unlike) {
            const WordNeighbours N = word_neighbours(lat, packing, pitch, Lx, Ly, W, helical, y, w, false);
            nA += __popc(N.v);
            n += __popc((N.v ^ N.nb[0]) & N.valid) + __popc((N.v ^ N.nb[2]) & N.valid);
            if (geometry == kTRI6) n += __popc((N.v ^ N.nb[4]) & N.valid);
        } else {
            nA += __popc(site_word(lat, packing, pitch, Lx, y, w));
        }
    }
    if (unlike) block_add(n, unlike);
    __syncthreads();
    if (sites_A) block_add(nA, sites_A);
}

// Fraction of first neighbours, random-neighbour estimator (sample m): the number
// of sites whose chosen nearest neighbour has the same type.  Site i's neighbour is
// direction floor(w z / 2^32) of (1,0), (-1,0), (0,1), (0,-1), (1,-1), (-1,1) (the
// first four for SQ4), w = word (i mod 4) of Philox(seed, {i div 4, 0xFFFFFFFE,
// m_lo, m_hi}); periodic wrap, or the helical wrap of x into the next row.
//
// A thread per 32-site word: the six comparisons are word operations, and the three
// bits of every site's direction are shifted into three planes that select among
// them.  Bound: the Philox blocks' wide multiplies, one block per four sites; a row
// whose first site is not a multiple of four takes a ninth block per word and a shift.
// 8192^2: 229 us with a thread per four sites, 74 us so.
__global__ void ffn_kernel(const void *lat, int packing, int Lx, int Ly, int pitch, int geometry, int helical,
                           uint32_t k0, uint32_t k1, unsigned long long m, long long *out)
{
    const uint32_t z = geometry == kTRI6 ? 6u : 4u;
    const int W = (Lx + 31) / 32;
    const long long nwords = (long long)W * Ly;
    long long n = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nwords;
         i += (long long)gridDim.x * blockDim.x) {
        const int y = (int)((uint32_t)i / (uint32_t)W), w = (int)((uint32_t)i - (uint32_t)y * (uint32_t)W);
        const uint32_t site = (uint32_t)y * (uint32_t)Lx + 32u * (uint32_t)w, off = site & 3u;
        uint32_t d0 = 0u, d1 = 0u, d2 = 0u;  // the directions' bits, site 4 (site / 4) at bit 0
        auto push = [&](uint32_t group, uint32_t &e0, uint32_t &e1, uint32_t &e2) {
            const Philox4 pw = philox4(group, 0xFFFFFFFEu, (uint32_t)m, (uint32_t)(m >> 32), k0, k1);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const uint32_t k = __umulhi(pw.v[r], z);
                e0 = __funnelshift_r(e0, k, 1);
                e1 = __funnelshift_r(e1, k >> 1, 1);
                e2 = __funnelshift_r(e2, k >> 2, 1);
            }
        };
        // the groups of four that hold the word's sites: 8, or 9, fewer in a row's last word
        // (4 x 200000: 12.8 us with 8 for every word, 8.0 so)
        const uint32_t groups = (off + (uint32_t)min(32, Lx - 32 * w) + 3u) >> 2;
        const uint32_t first8 = min(groups, 8u);
#pragma unroll 2
        for (uint32_t g = 0; g < first8; ++g) push((site >> 2) + g, d0, d1, d2);
        if (first8 < 8u) {
            d0 >>= 32u - 4u * first8;
            d1 >>= 32u - 4u * first8;
            d2 >>= 32u - 4u * first8;
        }
        if (off != 0u) {
            uint32_t h0 = 0u, h1 = 0u, h2 = 0u;  // four more, in the top bits
            if (groups > 8u) push((site >> 2) + 8u, h0, h1, h2);
            d0 = __funnelshift_r(d0, h0 >> 28, off);
            d1 = __funnelshift_r(d1, h1 >> 28, off);
            d2 = __funnelshift_r(d2, h2 >> 28, off);
        }
        const WordNeighbours N = word_neighbours(lat, packing, pitch, Lx, Ly, W, helical, y, w, true);
        // the chosen neighbour: direction = 4 d2 + 2 d1 + d0
        const uint32_t c01 = (d0 & N.nb[1]) | (~d0 & N.nb[0]), c23 = (d0 & N.nb[3]) | (~d0 & N.nb[2]);
        const uint32_t c45 = (d0 & N.nb[5]) | (~d0 & N.nb[4]);
        const uint32_t c = (d2 & c45) | (~d2 & ((d1 & c23) | (~d1 & c01)));
        n += __popc(~(N.v ^ c) & N.valid);
    }
    block_add(n, out);
}

// One byte per site (nonzero = A) into the bit store: a thread per 32-site word, its bytes
// read as the nine aligned words that hold them (byte by byte at the buffer's ends).  8192^2: 161 us with a lane per byte, 14 us so.
__device__ __forceinline__ uint32_t packed_word(const uint8_t *bytes, long long N, long long at, int n)
{
    const uint8_t *const from = bytes + at;
    const uint32_t sh = 8u * (uint32_t)((uintptr_t)from & 3u);
    uint32_t v = 0u;
    if (n == 32 && at >= 4 && at + 36 <= N) {
        const uint32_t *const p = (const uint32_t *)((uintptr_t)from & ~(uintptr_t)3);
        if (((uintptr_t)from & 15u) == 0u) {
            return nonzero_bytes(((const uint4 *)from)[0]) | (nonzero_bytes(((const uint4 *)from)[1]) << 16);
        }
        uint32_t lo = p[0];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const uint32_t hi = p[q + 1];
            v |= nonzero_bytes(__funnelshift_r(lo, hi, sh)) << (4 * q);
            lo = hi;
        }
        return v;
    }
    for (int b = 0; b < n; ++b) v |= (from[b] ? 1u : 0u) << b;
    return v;
}

__global__ void pack_kernel(const uint8_t *bytes, void *lat, int packing, int Lx, int Ly, int pitch)
{
    const long long N = (long long)Lx * Ly;
    const int W = (Lx + 31) / 32;
    const long long nwords = (long long)W * Ly;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nwords;
         i += (long long)gridDim.x * blockDim.x) {
        const int y = (int)((uint32_t)i / (uint32_t)W), w = (int)((uint32_t)i - (uint32_t)y * (uint32_t)W);
        const int n = min(32, Lx - 32 * w);
        const uint32_t v = packed_word(bytes, N, (long long)y * Lx + 32 * w, n);
        if (packing == kPackBit) {
            ((uint32_t *)lat)[(size_t)y * pitch + w] = v;
            continue;
        }
        uint8_t *const row = (uint8_t *)lat + (size_t)y * pitch + 32 * w;
        if ((((uintptr_t)row) & 3u) == 0u) {
            for (int q = 0; 4 * q < n; ++q) ((uint32_t *)row)[q] = spread_bits(v >> (4 * q));
        } else {
            for (int b = 0; b < n; ++b) row[b] = (uint8_t)((v >> b) & 1u);
        }
    }
}

// One byte per site from the store: a thread per 16 bytes of output (100^2 with its copy and
// wait: 16.3 us; site by site where a row ends among the 16, 17.9).
__global__ void unpack_kernel(const void *lat, int packing, int Lx, int Ly, int pitch, uint8_t *bytes)
{
    const long long N = (long long)Lx * Ly;
    const long long parts = (N + 15) / 16;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < parts;
         t += (long long)gridDim.x * blockDim.x) {
        const uint32_t i = 16u * (uint32_t)t;
        int y = (int)(i / (uint32_t)Lx), x = (int)(i - (uint32_t)y * (uint32_t)Lx);
        const int n = (int)min(16ll, N - (long long)i);
        uint32_t v = 0u;
        for (int b = 0; b < n;) {  // the rows' parts: one, two, or more of rows below 16 sites
            const int take = min(n - b, Lx - x);
            uint32_t part = 0u;
            if (packing == kPackBit) {
                const uint32_t *const row = (const uint32_t *)lat + (size_t)y * pitch;
                const int w = x >> 5, s = x & 31;
                part = s + take <= 32 ? row[w] >> s : __funnelshift_r(row[w], row[w + 1], s);
            } else {
                const uint8_t *const row = (const uint8_t *)lat + (size_t)y * pitch + x;
                const int lead = (int)((uintptr_t)row & 3u);
                if (((uintptr_t)lat & 3u) == 0u && (pitch & 3) == 0) {
                    const uint32_t *const words = (const uint32_t *)(row - lead);
                    uint32_t in[5];  // the last word is still within the row's padding
#pragma unroll
                    for (int q = 0; q < 5; ++q) in[q] = 4 * q < lead + take ? words[q] : 0u;
#pragma unroll
                    for (int q = 0; q < 4; ++q) part |= nonzero_bytes(__funnelshift_r(in[q], in[q + 1], 8 * lead)) << (4 * q);
                } else {
                    for (int k = 0; k < take; ++k) part |= (row[k] ? 1u : 0u) << k;
                }
            }
            v |= (part & ((1u << take) - 1u)) << b;
            b += take;
            x = 0;
            ++y;
        }
        if (n == 16 && (((uintptr_t)bytes) & 15u) == 0u) {
            ((uint4 *)bytes)[t] = make_uint4(spread_bits(v), spread_bits(v >> 4), spread_bits(v >> 8), spread_bits(v >> 12));
        } else {
            for (int b = 0; b < n; ++b) bytes[(size_t)i + b] = (uint8_t)((v >> b) & 1u);
        }
    }
}

int grid_for(long long work, int per_block)
{
    long long g = (work + per_block - 1) / per_block;
    if (g < 1) g = 1;
    if (g > 152 * 16) g = 152 * 16;
    return (int)g;
}

}  // namespace

size_t init_scratch_bytes() { return 2080; }
static_assert(sizeof(SelectState) <= 2080, "placement scratch");

cudaError_t launch_init_lattice(void *lat, size_t lat_bytes, int packing, int Lx, int Ly, int pitch, uint32_t key0,
                                uint32_t key1, long long nA, void *scratch, cudaStream_t stream)
{
    const long long N = (long long)Lx * Ly;
    SelectState *st = (SelectState *)scratch;
    int mode = 2;
    if (nA <= 0) mode = 0;
    else if (nA >= N) mode = 1;
    if (mode == 2) {
        // Rank nA: the last A site among all keys.  After log2(N) + 8 bits the bucket holds
        // more than the site with a chance of 2^-8; the last pass finishes then.  The store
        // is still zero here: it holds the counts of 12-bit digits (and is left zero).
        select_start_kernel<<<1, kBlock, 0, stream>>>(st, nA);
        const int g = grid_for(N, kBlock * 8);
        const bool wide = lat_bytes >= 4096 * sizeof(unsigned int) && ((uintptr_t)lat & 3u) == 0u;
        int need = 8;
        while ((1ll << (need - 8)) < N) ++need;
        // The first pass counts every site: 8 bits of it keep the CTAs' counts few, and 12
        // save a pass where a pass is long.  The others count a bucket's sites.
        for (int have = 0; have < need;) {
            const int bits = wide && (have > 0 || N >= (1ll << 24)) ? 12 : 8;
            have += bits;
            if (bits == 12) select_kernel<12><<<g, kBlock, 0, stream>>>(N, key0, key1, st, (unsigned int *)lat, have >= need);
            else select_kernel<8><<<g, kBlock, 0, stream>>>(N, key0, key1, st, st->hist, have >= need);
        }
    }
    const int g = grid_for(N, kBlock);
    mark_kernel<<<g, kBlock, 0, stream>>>(lat, packing, Lx, Ly, pitch, key0, key1, mode, st);
    return cudaGetLastError();
}

cudaError_t launch_tally(const void *lat, int packing, int Lx, int Ly, int pitch, int geometry, int helical,
                         long long *unlike, long long *sites_A, cudaStream_t stream)
{
    const long long nwords = (long long)((Lx + 31) / 32) * Ly;
    tally_kernel<<<grid_for(nwords, kBlock * 2), kBlock, 0, stream>>>(lat, packing, Lx, Ly, pitch, geometry, helical,
                                                                    unlike, sites_A);
    return cudaGetLastError();
}

cudaError_t launch_recount(const void *lat, int packing, int Lx, int Ly, int pitch, int geometry,
                           long long *out, cudaStream_t stream, int helical)
{
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(long long), stream);
    if (e != cudaSuccess) return e;
    return launch_tally(lat, packing, Lx, Ly, pitch, geometry, helical, out, nullptr, stream);
}

cudaError_t launch_ffn(const void *lat, int packing, int Lx, int Ly, int pitch, int geometry, int helical,
                       uint32_t key0, uint32_t key1, long long sample, long long *out, cudaStream_t stream)
{
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(long long), stream);
    if (e != cudaSuccess) return e;
    const long long nwords = (long long)((Lx + 31) / 32) * Ly;
    ffn_kernel<<<grid_for(nwords, kBlock), kBlock, 0, stream>>>(lat, packing, Lx, Ly, pitch, geometry, helical,
                                                              key0, key1, (unsigned long long)sample, out);
    return cudaGetLastError();
}

cudaError_t launch_pack(const uint8_t *bytes, void *lat, int packing, int Lx, int Ly, int pitch,
                        cudaStream_t stream)
{
    const long long nwords = (long long)((Lx + 31) / 32) * Ly;
    pack_kernel<<<grid_for(nwords, kBlock), kBlock, 0, stream>>>(bytes, lat, packing, Lx, Ly, pitch);
    return cudaGetLastError();
}

cudaError_t launch_unpack(const void *lat, int packing, int Lx, int Ly, int pitch, uint8_t *bytes,
                          cudaStream_t stream)
{
    const long long N = (long long)Lx * Ly;
    unpack_kernel<<<grid_for((N + 15) / 16, kBlock), kBlock, 0, stream>>>(lat, packing, Lx, Ly, pitch, bytes);
    return cudaGetLastError();
}

}  // namespace klmc
