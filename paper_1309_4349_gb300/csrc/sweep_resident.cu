// sweep_resident.cu -- Kawasaki exchange sweeps with the lattice resident in shared
// memory for the whole launch (section "Massive Parallel Kawasaki Kinetics": every
// iteration performs one exchange per domain of a random decomposition, all in
// parallel; here the decomposition is a conflict-free shifted sublattice phase).
//
// Work split.  One lattice per thread-block cluster of C CTAs (C = 1 is a plain
// CTA).  CTA c of the cluster owns the row band [Y_c, Y_c+1), Y_c = floor(c Ly / C),
// and keeps band rows plus two halo rows on each side in shared memory: local row
// lr holds global row (Y_c - 2 + lr) mod Ly.  A phase's anchor rows are split by
// band; every read of an anchor's neighbourhood (rows y-2 .. y+2) is local.  An
// accepted exchange flips its two sites in every copy of their rows: the local
// copy and, for rows within two of a band edge, the copies held by the
// neighbouring CTAs, through distributed shared memory.  Phases are separated by
// a cluster barrier (release/acquire), so the next phase sees every flip.
//
// Phase blocks.  When the bands are tall enough, a cluster of C > 1 CTAs instead
// advances K consecutive phases (K = 2 or 4) between exchanges.  Each CTA
// keeps D = 2K + 1 halo rows on each side, and in the j-th phase of a block
// evaluates every anchor within 2 (K - 1 - j) + 1 rows of its band: a site's new
// value depends only on sites at most two rows away, so after K phases the band
// is exact although the outer halo rows are not.  The anchors outside the band
// are evaluated again by the CTA that owns them, with the same counter-based
// random numbers, hence identical results; only anchors of the own band are
// counted.  All flips are local.  At the end of a block each CTA stores its D
// lowest and D highest band rows into mailboxes in the neighbouring CTAs'
// shared memory (double-buffered by block parity) and waits for its own two
// neighbours' rows, which it copies into its halo rows.
//
// Row layout.  A shared-memory row is W words of 32 sites at a stride of RW = W + 2
// words, the bits of the last word past the row's end zero.  The windows of the
// words at a row's ends reach around them (WordEnds in sweep_common.cuh).
//
// Evaluation.  One thread handles the anchors of one 32-site word of one anchor
// row.  Neighbour comparisons of all 32 positions are bitwise operations summed by
// carry-save adders into bit planes of S, the like ones among the six neighbours
// that only one site of an unlike pair touches.  Its
// exchange changes the number of unlike contacts by dn = 2 (S - 3).  Unlike
// pairs whose S lies in the draw range draw a Philox number; the rest are accepted
// outright (Metropolis acceptance min{1, exp(-omega dn / kT)}, steps a-c).  A
// lane draws for its own anchors, two Philox evaluations interleaved at a time:
// a phase is short, so its cost is the latency of its slowest task.
#include <string.h>

#include <type_traits>

#include "klmc_internal.h"
#include "philox.cuh"

namespace klmc {
namespace {

#include "sweep_common.cuh"
#include "cluster_exchange.cuh"

// XOR v into the 32-bit word at shared address addr of CTA `rank` of the cluster.
__device__ __forceinline__ void xor_word(uint32_t addr, uint32_t rank, bool local, uint32_t v)
{
    if (v == 0u) return;
    if (local) {
        asm volatile("red.shared.xor.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
    } else {
        uint32_t remote;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(rank));
        asm volatile("red.shared::cluster.xor.b32 [%0], %1;" ::"r"(remote), "r"(v) : "memory");
    }
}

// XOR v into the 32-bit word at shared address addr of this CTA, unconditionally.
__device__ __forceinline__ void red_xor_local(uint32_t addr, uint32_t v)
{
    asm volatile("red.shared.xor.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

struct Acc {
    uint32_t unl, drw, acc;
    int32_t dn;  // n_unlike change / 2
};

struct Geo {
    int Lx, Ly, W, RW;
    uint32_t magicW, one;  // task t is word t - m W of row m = (t magicW) >> 32 (W = 1: magicW 0, one ~0, m = t)
    uint32_t k0, k1;
    bool tri;            // triangular (else square) geometry
    int sign;            // draw when the exchange raises (+1) / lowers (-1) E; 0: never
    int C, rank, Y0, Y1;
    int prevY, prevH;    // band of CTA rank-1 (mod C)
    int nextY, nextH;    // band of CTA rank+1 (mod C)
    uint32_t lat_addr;   // shared address of local row 0
    int D;               // halo rows on each side: local row lr holds row (Y0 - D + lr) mod Ly
    int base;            // (Y0 - D) mod Ly
    int tabW;            // words of a table's anchor masks (even)
    int nlast;           // sites of a row's last word
    uint32_t magicInner;  // as magicW for the words of a row without its kEndCount end words (band kernel)
};

__device__ __forceinline__ int task_row(const Geo &g, int t)
{
    return (int)(__umulhi((uint32_t)t, g.magicW) + ((uint32_t)t & g.one));
}

// Flips, in this CTA's rows, the accepted anchors acc of the word at shared address wa
// and their partners.  Atomics of 0 cost less than branches around them.
template <int OI, Windows WN = kEnds>
__device__ __forceinline__ void flip_pairs(uint32_t wa, int RW, const WordEnds &E, uint32_t acc)
{
    const uint32_t rowbytes = 4u * (uint32_t)RW;
    const uint32_t wb = OI == 0 ? wa : (OI == 1 ? wa + rowbytes : wa - rowbytes);
    uint32_t b;
    const uint32_t next = partners<OI, WN>(acc, E, b);
    if (OI == 0) {
        red_xor_local(wa, acc | b);
    } else {
        red_xor_local(wa, acc);
        red_xor_local(wb, b);
    }
    if (OI != 1) red_xor_local(WN == kPlain ? wb + 4u : wb + 4u * (uint32_t)E.r, next);
}

// Flips m in word j of global row r (unwrapped, in [Y0 - 1, Y1]) in every CTA holding a copy.
__device__ __forceinline__ void flip_global_row(const Geo &g, int r, int j, uint32_t m)
{
    if (m == 0u) return;
    const uint32_t word = g.lat_addr + 4u * (uint32_t)j, rowbytes = 4u * (uint32_t)g.RW;
    const int lr_self = r - g.Y0 + 2;
    if (lr_self >= 4 && lr_self < g.Y1 - g.Y0) {  // interior row: local copy only
        red_xor_local(word + rowbytes * (uint32_t)lr_self, m);
        return;
    }
    const int gr = r < 0 ? r + g.Ly : (r >= g.Ly ? r - g.Ly : r);
    if (g.C == 1) {  // rows 0, 1 and Ly-2, Ly-1 also live in the opposite halo
        for (int lr = gr + 2 >= g.Ly ? gr + 2 - g.Ly : gr + 2; lr < g.Ly + 4; lr += g.Ly)
            red_xor_local(word + rowbytes * (uint32_t)lr, m);
        return;
    }
    for (int k = 0; k < 3; ++k) {
        if (k == 2 && g.C == 2) break;  // both neighbours are the same CTA
        const int d = k == 0 ? (g.rank == 0 ? g.C - 1 : g.rank - 1)
                             : (k == 1 ? g.rank : (g.rank + 1 == g.C ? 0 : g.rank + 1));
        const int Yd = k == 0 ? g.prevY : (k == 1 ? g.Y0 : g.nextY);
        const int Hd = k == 0 ? g.prevH : (k == 1 ? g.Y1 - g.Y0 : g.nextH);
        int lr = gr - Yd + 2;
        if (lr < 0) lr += g.Ly;
        if (lr >= g.Ly) lr -= g.Ly;
        for (; lr < Hd + 4; lr += g.Ly) xor_word(word + rowbytes * (uint32_t)lr, (uint32_t)d, d == g.rank, m);
    }
}

// Barrier of the CTA's first NT threads, which run the tasks.
template <int NT>
__device__ __forceinline__ void task_barrier()
{
    asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
}

// Barrier of the whole CTA, reached by different warps in different places.
__device__ __forceinline__ void cta_barrier() { asm volatile("bar.sync 0;" ::: "memory"); }

// Per-phase task table: the anchor mask of every word and, per task row mi, the
// local row and the row's first site index, so that a task loads two entries
// instead of recomputing them.  The resident kernel keeps two chunks of kChunk phases
// (the current one and the next), the band kernel the phases of its block.
constexpr int kChunk = 4;

struct TaskTab {  // a table's storage and capacity
    uint32_t *am;
    int2 *row;   // (local row, y * Lx)
    int maxw, maxrows;
};

__device__ __forceinline__ bool table_fits(const Geo &g, const PhaseR &P, const TaskTab &T)
{
    return g.W <= T.maxw && P.c[3] <= T.maxrows;
}

// Fills the table entries with index = lane0 mod step, so that a warp (step 32) or a
// CTA (step THREADS) builds it together.  The table holds the phase's words and rows.
template <bool BLOCKED>
__device__ __forceinline__ void build_task_table(const PhaseR &P, const Geo &g, const TaskTab &T, int lane0,
                                                 int step)
{
    for (int j = lane0; j < g.W; j += step) T.am[j] = anchor_mask(j << 5, P, g.Lx);
    for (int mi = lane0; mi < P.c[3]; mi += step) {
        const int m = mi < P.c[0] ? P.a[0] + mi
                    : (mi < P.c[1] ? P.a[1] + mi : (mi < P.c[2] ? P.a[2] + mi : P.a[3] + mi));
        int y = P.ry + P.py * m;
        if (y >= g.Ly) y -= g.Ly;
        int lr;
        if (BLOCKED) {
            lr = y - g.base;
            if (lr < 0) lr += g.Ly;
        } else {
            lr = y - g.Y0 + 2;
        }
        T.row[mi] = make_int2(lr, y * g.Lx);
    }
}

// What a phase's tasks need of its schedule entry, prepared with the task table.
struct __align__(16) PhaseHdr {
    int nlane;        // lanes with tasks: the phase's words, each split over 2^ls lanes
    int code;         // orientation + 4 ls
    uint32_t hk, la;  // the phase's part of the draw key
};

// Lanes per word (log2) of a phase of ntask words on NT threads.  A split word's
// lanes all evaluate it and each keeps the anchors of its part, which divides the
// draws (the longest step of a lane) among them.  With 480 task threads the split ends
// at 192 lanes: more lanes than that cost every scheduler a warp that shares no draws
// (300^2 on 16 CTAs 1.01 -> 0.99 us per phase, 256^2 0.96 -> 0.95).
template <int NT>
__device__ __forceinline__ int word_split(int ntask)
{
    constexpr int kLanes = NT > 256 ? 192 : NT;
    return 4 * ntask <= kLanes ? 2 : (2 * ntask <= kLanes ? 1 : 0);
}

// One task of a phase: the word at p of an anchor row in local row lr (word j of it),
// the site index of its first site, its ends and its anchors.
struct Task {
    const uint32_t *p;
    int j, lr;
    uint32_t site, am;
    WordEnds E;
};

template <bool BLOCKED>
__device__ __forceinline__ Task load_task(const uint32_t *lat, const Geo &g, int tl, int ls, const PhaseR &P,
                                          bool use_tab, const uint32_t *tab)
{
    Task k;
    const int t = tl >> ls;
    const int mi = task_row(g, t);
    k.j = t - mi * g.W;
    int ybase;
    if (use_tab) {
        k.am = tab[k.j];
        const int2 r = *(const int2 *)(tab + g.tabW + 2 * mi);
        k.lr = r.x;
        ybase = r.y;
    } else {
        const int m = mi < P.c[0] ? P.a[0] + mi
                    : (mi < P.c[1] ? P.a[1] + mi : (mi < P.c[2] ? P.a[2] + mi : P.a[3] + mi));
        int y = P.ry + P.py * m;
        if (y >= g.Ly) y -= g.Ly;
        if (BLOCKED) {
            k.lr = y - g.base;
            if (k.lr < 0) k.lr += g.Ly;
        } else {
            k.lr = y - g.Y0 + 2;  // y is a band row
        }
        ybase = y * g.Lx;
        k.am = anchor_mask(k.j << 5, P, g.Lx);
    }
    // a split word's part (the thread count is a multiple of 4, so a thread's part is fixed)
    const int bits = 32 >> ls;
    k.am &= (0xFFFFFFFFu >> (32 - bits)) << ((tl & ((1 << ls) - 1)) * bits);
    k.site = (uint32_t)(ybase + (k.j << 5));
    k.p = lat + k.lr * g.RW + k.j;
    k.E = word_ends(k.j, g.W, g.nlast, 0);
    return k;
}

// One phase of one band, by the first NT threads of the CTA, the thread's first task
// already loaded.  Every task is (anchor row, word j).  BLOCKED: the anchors span the
// band and part of its halo, all flips are local, and only anchors of the band are
// counted; otherwise the anchors are those of the band and flips reach every copy of
// their rows.
//
// Bound: a warp issues an instruction about every five cycles (dependent operations
// of one or two warps per scheduler), so a phase lasts as long as the instruction
// stream of its busiest warp.  Branches in it cost most: the geometry, the orientation
// and the rare row shapes are template parameters.
template <int G, int OI, int NT, bool BLOCKED, Windows WN>
__device__ __forceinline__ void run_phase(const uint32_t *lat, const Geo &g, const PhaseHdr &h, Task k,
                                          const PhaseR &P, const DrawThr &T, const DrawKey &dk, Acc &A,
                                          bool use_tab, const uint32_t *tab)
{
    // b = a + o: (1,0) -> same row, +1; (0,1) -> next row; (1,-1) -> previous row, +1
    constexpr int bdy = OI == 0 ? 0 : (OI == 1 ? 1 : -1);
    const int H = g.Y1 - g.Y0;
    for (int tl = threadIdx.x; tl < h.nlane;) {
        uint32_t ta, tb;
        Planes S;
        evaluate<G, OI, WN>(k.p, g.RW, k.E, ta, tb, S);
        const uint32_t unl = (ta ^ tb) & k.am;
        const uint32_t dmask = unl & draw_positions(S, g.sign);
        const uint32_t acc = (unl & ~dmask) | draw_accepts(dmask, S, k.site, dk, T);
        const uint32_t own = !BLOCKED || (unsigned)(k.lr - g.D) < (unsigned)H ? ~0u : 0u;
        const uint32_t oacc = acc & own;
        const int na = __popc(oacc);
        A.unl += __popc(unl & own);
        A.drw += __popc(dmask & own);
        A.acc += na;
        A.dn += half_dn(S, oacc, na);
        // One CTA: rows 2 .. Ly-3 have no copy in a halo.
        if (BLOCKED || (g.C == 1 && k.lr >= 5 && k.lr < H - 1)) {
            flip_pairs<OI>(smem_addr(k.p), g.RW, k.E, acc);
        } else {
            const int yu = k.lr - g.D + g.Y0;  // unwrapped band row
            uint32_t b;
            const uint32_t next = partners<OI>(acc, k.E, b);
            flip_global_row(g, yu, k.j, acc);
            flip_global_row(g, yu + bdy, k.j, b);
            flip_global_row(g, yu + bdy, k.j + k.E.r, next);
        }
        tl += NT;
        if (tl < h.nlane) k = load_task<BLOCKED>(lat, g, tl, h.code >> 2, P, use_tab, tab);
    }
}

// Band kernel: one phase with two tasks per lane (t and t + THREADS) sharing one
// pass of the warp's draw queue.  Blocked (all flips local, only the band's anchors
// counted), with the phase's task table when it fits.
struct TaskPrep {
    uint32_t dmask, acc;  // positions that need a draw; accepted without one
    Planes S;
    uint32_t base;        // site index of position 0
    int lr, j;
    bool own;
};

// Which words of the anchor rows a loop of tasks takes: all, those away from the rows' ends
// (plain windows), or the first and the last two.
enum RowPart { kAllWords, kInnerWords, kEndWords };
constexpr int kEndCount = 3;

template <int G, int OI, RowPart RP>
__device__ __forceinline__ void band_task_prep(const uint32_t *lat, const Geo &g, const PhaseR &P, bool use_tab,
                                               const TaskTab *tt, int t, bool valid, TaskPrep &T, Acc &A)
{
    constexpr Windows WN = RP == kInnerWords ? kPlain : kFix;
    uint32_t am = 0u, ta = 0u, tb = 0u;
    Planes S = {0u, 0u, 0u};
    int ybase = 0, j = 0, lr = 0;
    if (valid) {
        int mi;
        if (RP == kInnerWords) {
            mi = (int)__umulhi((uint32_t)t, g.magicInner);
            j = t - mi * (g.W - kEndCount) + 1;
        } else if (RP == kEndWords) {
            mi = t / kEndCount;
            j = t - mi * kEndCount;
            j = j == 0 ? 0 : g.W - kEndCount + j;
        } else {
            mi = task_row(g, t);
            j = t - mi * g.W;
        }
        if (use_tab) {
            const int2 r = tt->row[mi];
            lr = r.x;
            ybase = r.y;
            am = tt->am[j];
        } else {
            const int m = mi < P.c[0] ? P.a[0] + mi
                        : (mi < P.c[1] ? P.a[1] + mi : (mi < P.c[2] ? P.a[2] + mi : P.a[3] + mi));
            int y = P.ry + P.py * m;
            if (y >= g.Ly) y -= g.Ly;
            lr = y - g.base;
            if (lr < 0) lr += g.Ly;
            ybase = y * g.Lx;
            am = anchor_mask(j << 5, P, g.Lx);
        }
        evaluate<G, OI, WN>(lat + lr * g.RW + j, g.RW, word_ends(j, g.W, g.nlast, 0), ta, tb, S);
    }
    const uint32_t unl = (ta ^ tb) & am;
    T.dmask = unl & draw_positions(S, g.sign);
    T.acc = unl & ~T.dmask;
    T.S = S;
    T.base = (uint32_t)(ybase + (j << 5));
    T.lr = lr;
    T.j = j;
    T.own = (unsigned)(lr - g.D) < (unsigned)(g.Y1 - g.Y0);
    if (T.own) {
        A.unl += __popc(unl);
        A.drw += __popc(T.dmask);
    }
}

template <int OI, RowPart RP>
__device__ __forceinline__ void band_task_finish(const Geo &g, const TaskPrep &T, uint32_t acc, Acc &A)
{
    if (!acc) return;
    if (T.own) {
        const int na = __popc(acc);
        A.acc += na;
        A.dn += half_dn(T.S, acc, na);
    }
    flip_pairs<OI, RP == kInnerWords ? kPlain : kFix>(g.lat_addr + 4u * (uint32_t)(T.lr * g.RW + T.j), g.RW, word_ends(T.j, g.W, g.nlast, 0), acc);
}

// INNER: wide rows.  Their words away from the ends need no distances around them (7% of
// a phase of 8192^2); the end words go first, to the last warps, which have the fewest
// others.
template <int G, int OI, int THREADS, bool INNER>
__device__ __forceinline__ void run_phase_pair(const uint32_t *lat, const Geo &g, const PhaseR &P,
                                               const DrawThr &T, int f, uint32_t s_lo, uint32_t s_hi,
                                               Acc &A, uint32_t *q, const TaskTab *tt, const uint32_t (&rk)[2][8])
{
    constexpr RowPart RP = INNER ? kInnerWords : kAllWords;
    const int lane = threadIdx.x & 31;
    const int ntask = INNER ? P.c[3] * (g.W - kEndCount) : P.ntask;
    const bool use_tab = tt != nullptr && table_fits(g, P, *tt);
    const DrawKey dk = draw_key((uint32_t)f, s_lo, s_hi, g.k0, g.k1);
    if (INNER) {
        for (int t = THREADS - 32 - (int)(threadIdx.x & ~31) + lane; t < kEndCount * P.c[3]; t += THREADS) {
            TaskPrep T0;
            band_task_prep<G, OI, kEndWords>(lat, g, P, use_tab, tt, t, true, T0, A);
            band_task_finish<OI, kEndWords>(g, T0, T0.acc | draw_accepts(T0.dmask, T0.S, T0.base, dk, T), A);
        }
        __syncwarp();
    }
    for (int t0 = threadIdx.x & ~31; t0 < ntask; t0 += 2 * THREADS) {
        const int ta = t0 + lane, tb = t0 + THREADS + lane;
        TaskPrep T0, T1;
        band_task_prep<G, OI, RP>(lat, g, P, use_tab, tt, ta, ta < ntask, T0, A);
        band_task_prep<G, OI, RP>(lat, g, P, use_tab, tt, tb, tb < ntask, T1, A);
        uint32_t a0, a1;
        draw_accepts_queue2(T0.dmask, T0.S, T0.base, T1.dmask, T1.S, T1.base, dk, rk, T, q, a0, a1);
        band_task_finish<OI, RP>(g, T0, T0.acc | a0, A);
        band_task_finish<OI, RP>(g, T1, T1.acc | a1, A);
    }
}

template <int G, int THREADS, bool INNER>
__device__ __forceinline__ void run_phase_pair_oi(const uint32_t *lat, const Geo &g, const PhaseR &P,
                                                  const DrawThr &T, int f, uint32_t s_lo, uint32_t s_hi,
                                                  Acc &A, uint32_t *q, const TaskTab *tt, const uint32_t (&rk)[2][8])
{
    if (P.oi == 0) run_phase_pair<G, 0, THREADS, INNER>(lat, g, P, T, f, s_lo, s_hi, A, q, tt, rk);
    else if (G == kTRI6 && P.oi == 2) run_phase_pair<G, 2, THREADS, INNER>(lat, g, P, T, f, s_lo, s_hi, A, q, tt, rk);
    else run_phase_pair<G, 1, THREADS, INNER>(lat, g, P, T, f, s_lo, s_hi, A, q, tt, rk);
}

// Rows of at least this many words have their end words apart.
constexpr int kInnerRowWords = 96;

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

__device__ __forceinline__ uint32_t cluster_nctarank()
{
    uint32_t v;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(v));
    return v;
}

__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t v;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(v));
    return v;
}

__device__ __forceinline__ uint32_t dynamic_smem_bytes()
{
    uint32_t v;
    asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(v));
    return v;
}

// Dynamic shared memory a CTA may use (the kernels' static arrays take under 6 KB).
constexpr int kResidentMaxSmem = 227 * 1024 - 6144;

#ifndef KLMC_MAX_BLOCK
#define KLMC_MAX_BLOCK 4
#endif
static_assert(KLMC_MAX_BLOCK == 1 || KLMC_MAX_BLOCK == 2 || KLMC_MAX_BLOCK == 4 || KLMC_MAX_BLOCK == 8,
              "a sweep's 8 phases are whole blocks");

// Phases per block for a lattice of Lx x Ly sites split over C CTAs: the largest K
// of 8, 4, 2 (at most KLMC_MAX_BLOCK) whose halo D = 2K + 1 fits in every band
// (twice, for C = 2, so that a CTA's rows never overlap themselves) and whose
// rows and mailboxes fit in shared memory; 1 (a cluster barrier per phase)
// otherwise.
__host__ __device__ __forceinline__ int block_phases(int Lx, int Ly, int C)
{
    if (C <= 1) return 1;
    const int hmin = Ly / C, hmax = (Ly + C - 1) / C;
    const long long RW = (Lx + 95) / 32;
    for (int K = KLMC_MAX_BLOCK; K >= 2; K >>= 1) {
        const int D = 2 * K + 1;
        if (D > hmin || (C == 2 && 2 * D > hmin)) continue;
        if (RW * (hmax + 6 * D) * 4 > kResidentMaxSmem) continue;
        return K;
    }
    return 1;
}

// Phase table of (sweep s, phase f): the band's anchors, widened for a block.
__device__ __forceinline__ void phase_table(const Geo &g, int K, long long s, int f, PhaseR *P)
{
    const int e = K > 1 ? 2 * (K - 1 - (f & (K - 1))) + 1 : 0;
    phase_ranges(g.tri ? kTRI6 : kSQ4, g.Lx, g.Ly, g.W, g.Y0 - e, g.Y1 + e, g.k0, g.k1, s, f, P);
}

// Words of the task tables of one phase, and of the two chunks' (see TaskTab): anchor
// masks of W words (even, so that the row entries stay aligned) and the rows.  They hold
// every phase: its anchor rows lie in at most hmax + 2 (2K - 1) rows (K = 1: hmax) and are
// at least two apart, around the lattice's end too, so there are at most (hmax + 4K) / 2.
__host__ __device__ __forceinline__ int phase_table_words(int W, int hmax, int K)
{
    return ((W + 1) & ~1) + 2 * ((hmax + 4 * K) / 2 + 2);
}
__host__ __device__ __forceinline__ long long chunk_table_words(int W, int hmax, int K)
{
    return 2ll * kChunk * phase_table_words(W, hmax, K);
}
// Words of a CTA's rows (and mailboxes), where the tables start.
__host__ __device__ __forceinline__ long long resident_row_words(int RW, int hmax, int K)
{
    return ((long long)RW * (K > 1 ? hmax + 6 * (2 * K + 1) : hmax + 4) + 1) & ~1ll;
}

// Schedule entry and draw key of phase f of sweep s.
template <int NT>
__device__ __forceinline__ void prepare_entry(const Geo &g, int K, long long s, int f, PhaseR *P,
                                              PhaseHdr *h)
{
    phase_table(g, K, s, f, P);
    const DrawKey dk = draw_key((uint32_t)f, (uint32_t)(unsigned long long)s, (uint32_t)((unsigned long long)s >> 32),
                                g.k0, g.k1);
    const int ls = word_split<NT>(P->ntask);
    h->nlane = P->ntask << ls;
    h->code = P->oi + 4 * ls;
    h->hk = dk.hk;
    h->la = dk.la;
}

template <int V>
using Const = std::integral_constant<int, V>;

// Preparing a phase (a Philox block, the anchor rows' ranges, the tables) takes one
// warp about 600 cycles, half a phase of a lattice spread over a cluster.  So
// with more than 128 threads the last warp does nothing else: it prepares the
// next kChunk phases while the others, which synchronise among themselves, run the
// current ones, and meets them once per chunk.  (Two or four such warps were no faster,
// and took warps from the tasks: 400^2 on 8 CTAs 1.55 us per phase with four, 1.39 with one.)
// With 128 threads (several CTAs per SM, every warp busy) each of the four warps
// prepares one phase of the next chunk before its own tasks.
template <int THREADS, int MINB>
__global__ void __launch_bounds__(THREADS, MINB)
resident_sweep_kernel(const SweepJob *__restrict__ jobs, const SweepCall *__restrict__ calls,
                      const int *__restrict__ job_map, const SweepJob job0, const SweepCall call0)
{
    constexpr int kWarps = THREADS / 32;
    constexpr int kAhead = THREADS > 128 ? 1 : 0;
    constexpr int NT = THREADS - 32 * kAhead;  // threads with tasks
    constexpr int kPrep = kAhead > 0 ? kAhead : kWarps;  // warps that prepare
    static_assert(kPrep <= kChunk && kChunk % kPrep == 0, "each preparing warp has kChunk / kPrep phases");
    extern __shared__ __align__(16) uint32_t lat[];
    __shared__ PhaseR pp[2][kChunk];
    __shared__ PhaseHdr hdr[2][kChunk];
    __shared__ long long red[5][kWarps];
    __shared__ __align__(8) unsigned long long xbar[kExchangeBars];

    const int C = (int)cluster_nctarank();
    const int rank = (int)cluster_ctarank();
    const int job = job_map ? job_map[blockIdx.x / C] : (int)blockIdx.x / C;
    const SweepJob &J = jobs ? jobs[job] : job0;
    const SweepCall Cl = calls ? calls[job] : call0;
    if (Cl.n_mcs <= 0) return;  // uniform over the cluster

    Geo g;
    g.Lx = J.Lx; g.Ly = J.Ly; g.W = J.W; g.RW = J.RW; g.magicW = g.W == 1 ? 0u : (uint32_t)J.magicW; g.one = g.W == 1 ? ~0u : 0u;
    g.nlast = g.Lx - 32 * (g.W - 1);
    g.k0 = J.key0; g.k1 = J.key1;
    // The host's draw range is [z, 2(z-1)] (omega > 0), [0, z-2] (omega < 0) or empty.
    g.sign = J.draw_lo > J.draw_hi ? 0 : (J.draw_lo == 0 ? -1 : 1);
    g.tri = J.geometry == kTRI6;
    g.C = C;
    g.rank = rank;
    g.Y0 = (int)(((long long)rank * g.Ly) / C);
    g.Y1 = (int)(((long long)(rank + 1) * g.Ly) / C);
    {
        const int pr = rank == 0 ? C - 1 : rank - 1, nr = rank + 1 == C ? 0 : rank + 1;
        g.prevY = (int)(((long long)pr * g.Ly) / C);
        g.prevH = (int)(((long long)(pr + 1) * g.Ly) / C) - g.prevY;
        g.nextY = (int)(((long long)nr * g.Ly) / C);
        g.nextH = (int)(((long long)(nr + 1) * g.Ly) / C) - g.nextY;
    }
    g.lat_addr = smem_addr(lat);
    const int K = block_phases(g.Lx, g.Ly, C);
    const bool blocked = K > 1;
    g.D = blocked ? 2 * K + 1 : 2;
    g.base = g.Y0 - g.D < 0 ? g.Y0 - g.D + g.Ly : g.Y0 - g.D;
    const int hmax = (g.Ly + C - 1) / C;
    const int tid = threadIdx.x;
    const int H = g.Y1 - g.Y0;
    const int NL = H + 2 * g.D;

    // Load band and halo rows into padded shared-memory rows.
    for (int idx = tid; idx < NL * g.RW; idx += THREADS) {
        const int lr = idx / g.RW, w = idx - lr * g.RW;
        int y = g.Y0 - g.D + lr;
        y %= g.Ly;
        if (y < 0) y += g.Ly;
        lat[idx] = w < g.W ? store_word(J.lat, J.packing, J.pitch, y, w, g.Lx) : 0u;
    }
    // The tables follow the rows where the launch's shared memory holds them.
    const int tab_words = phase_table_words(g.W, hmax, K);
    uint32_t *const tab_base = lat + resident_row_words(g.RW, hmax, K);
    const bool tables = 4 * (resident_row_words(g.RW, hmax, K) + chunk_table_words(g.W, hmax, K)) <=
                        (long long)dynamic_smem_bytes();
    const int warp = tid >> 5, lane = tid & 31;
    const bool ahead_warp = kAhead > 0 && warp >= kWarps - kAhead;
    const DrawThr T = draw_thresholds(J);
    g.tabW = (g.W + 1) & ~1;
    unsigned long long t_att = 0, t_unl = 0, t_drw = 0, t_acc = 0;
    long long t_dn = 0;
    // Prepares chunk c (sweep c / 2, its phases kChunk (c & 1) ..) into buffer c & 1.
    auto prepare_chunk = [&](long long c) {
        const int buf = (int)(c & 1), f0 = kChunk * buf;
        const long long s = Cl.sweep0 + (c >> 1);
        if (kAhead > 0 && !ahead_warp) return;
        constexpr int kPer = kChunk / kPrep;
        const int q0 = (warp - (kWarps - kPrep)) * kPer;
        if (lane < kPer) {
            PhaseR *const P = &pp[buf][q0 + lane];
            prepare_entry<NT>(g, K, s, f0 + q0 + lane, P, &hdr[buf][q0 + lane]);
            if (rank == 0) t_att += (unsigned long long)P->att;  // the whole lattice's, counted once
        }
        __syncwarp();
        if (!tables) return;
#pragma unroll 1
        for (int q = q0; q < q0 + kPer; ++q) {
            const PhaseR P = pp[buf][q];
            uint32_t *const t = tab_base + (buf * kChunk + q) * tab_words;
            const TaskTab tt = {t, (int2 *)(t + g.tabW), g.W, (tab_words - g.tabW) / 2};
            if (blocked) build_task_table<true>(P, g, tt, lane, 32);
            else build_task_table<false>(P, g, tt, lane, 32);
        }
    };
    prepare_chunk(0);
    exchange_init(xbar);
    // Every CTA of the cluster must be running before any peer writes into it.
    if (C > 1) cluster_barrier();
    else cta_barrier();

    // Start energy for the trace, read before any CTA of this lattice can finish.
    const long long n_unlike0 = (tid == 0 && rank == 0 && Cl.trace_every > 0) ? J.state[kNUnlike] : 0;
    // The preparing warps: the next chunk's tables while the current one runs, then the
    // chunk's last barrier (every phase is a cluster barrier when bands are too thin
    // for blocks).
    Exchange X = exchange_for<NT>(xbar, g.lat_addr, C, rank, g.D * g.RW, J.copy_shortfall != 0);
    auto run_tasks = [&](auto geometry, auto is_blocked, auto has_fix) {
        constexpr int G = decltype(geometry)::value;
        constexpr bool BLOCKED = decltype(is_blocked)::value;
        constexpr Windows WN = decltype(has_fix)::value ? kFix : kEnds;
        int block = 0;
        for (long long it = 0; it < Cl.n_mcs; ++it) {
            const bool last = it + 1 == Cl.n_mcs;
            const long long s = Cl.sweep0 + it;
            DrawKey dk = draw_key(0u, (uint32_t)(unsigned long long)s, (uint32_t)((unsigned long long)s >> 32), g.k0,
                                  g.k1);
            Acc A = {0u, 0u, 0u, 0};
#pragma unroll 1
            for (int buf = 0; buf < 8 / kChunk; ++buf) {
                if (kAhead == 0 && !(last && buf == 1)) prepare_chunk(2 * it + buf + 1);
                const PhaseHdr *hp = hdr[buf];
                const uint32_t *tab = tab_base + buf * kChunk * tab_words;
                PhaseHdr h = hp[0];
                Task k = {};
                if (tid < h.nlane) k = load_task<BLOCKED>(lat, g, tid, h.code >> 2, pp[buf][0], tables, tab);
#pragma unroll 1
                for (int q = 0; q < kChunk; ++q) {
                    dk.hk = h.hk;
                    dk.la = h.la;
                    const int oi = h.code & 3;
                    const PhaseR &P = pp[buf][q];
                    if (oi == 0) run_phase<G, 0, NT, BLOCKED, WN>(lat, g, h, k, P, T, dk, A, tables, tab);
                    else if (G == kSQ4 || oi == 1) run_phase<G, 1, NT, BLOCKED, WN>(lat, g, h, k, P, T, dk, A, tables, tab);
                    else run_phase<G, 2, NT, BLOCKED, WN>(lat, g, h, k, P, T, dk, A, tables, tab);
                    if (q < kChunk - 1) {  // the next phase's entry does not wait for this one
                        tab += tab_words;
                        h = hp[q + 1];
                        if (tid < h.nlane) k = load_task<BLOCKED>(lat, g, tid, h.code >> 2, pp[buf][q + 1], tables, tab);
                    }
                    if (!BLOCKED && C > 1) {
                        cluster_barrier();
                        continue;
                    }
                    // Blocks of K phases end with an exchange, except the launch's last.  (One of
                    // more than kChunk phases ends in a later chunk than it began.)
                    const int ran = (KLMC_MAX_BLOCK > kChunk ? kChunk * buf : 0) + q + 1;
                    if (BLOCKED && (ran & (K - 1)) == 0 && !(last && buf == 1 && q == kChunk - 1)) {
                        task_barrier<NT>();
                        exchange_halos<NT>(lat, g.lat_addr, g.RW, g.Y1 - g.Y0, g.D, hmax, block++, X);
                    }
                    if (q == kChunk - 1) cta_barrier();
                    else task_barrier<NT>();
                }
            }
            t_unl += A.unl; t_drw += A.drw; t_acc += A.acc;
            t_dn += 2 * A.dn;
            // Energy trace: each CTA adds its cumulative dn; CTA 0 adds the start value
            // (the launcher zeroes the trace buffer).
            if (Cl.trace_every > 0 && (it + 1) % Cl.trace_every == 0) {
                const long long ws = warp_sum(t_dn);
                if (lane == 0 && ws != 0)
                    atomicAdd((unsigned long long *)&Cl.trace[(it + 1) / Cl.trace_every - 1],
                              (unsigned long long)ws);
                if (tid == 0 && rank == 0)
                    atomicAdd((unsigned long long *)&Cl.trace[(it + 1) / Cl.trace_every - 1],
                              (unsigned long long)n_unlike0);
            }
        }
    };
    if (ahead_warp) {
        for (long long c = 1; c <= 2 * Cl.n_mcs; ++c) {
            if (c < 2 * Cl.n_mcs) prepare_chunk(c);
            if (blocked || C == 1) {
                cta_barrier();
            } else {
                for (int q = 0; q < kChunk; ++q) cluster_barrier();
            }
        }
    } else if (blocked) {
        // (rows whose last word holds one site take a longer window: their own copy)
        if (g.nlast == 1) {
            if (g.tri) run_tasks(Const<kTRI6>{}, std::true_type{}, std::true_type{});
            else run_tasks(Const<kSQ4>{}, std::true_type{}, std::true_type{});
        } else {
            if (g.tri) run_tasks(Const<kTRI6>{}, std::true_type{}, std::false_type{});
            else run_tasks(Const<kSQ4>{}, std::true_type{}, std::false_type{});
        }
    } else {
        if (g.tri) run_tasks(Const<kTRI6>{}, std::false_type{}, std::true_type{});
        else run_tasks(Const<kSQ4>{}, std::false_type{}, std::true_type{});
    }
    if (blocked) exchange_end(X, J.copy_shortfall != 0, J.state);

    // Write the band back (main positions only).
    for (int idx = tid; idx < H * g.W; idx += THREADS) {
        const int r = idx / g.W, w = idx - r * g.W;
        const int y = g.Y0 + r;
        write_word(J.lat, J.packing, J.pitch, y, w, g.Lx, lat[(r + g.D) * g.RW + w]);
    }

    // Counters and energy.
    long long vals[5] = {(long long)t_att, (long long)t_unl, (long long)t_drw, (long long)t_acc, t_dn};
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const long long ws = warp_sum(vals[k]);
        if ((tid & 31) == 0) red[k][tid >> 5] = ws;
    }
    __syncthreads();
    if (tid < 5) {
        long long sum = 0;
        for (int w = 0; w < kWarps; ++w) sum += red[tid][w];
        const int slot = tid == 4 ? kNUnlike : kAttempts + tid;
        atomicAdd((unsigned long long *)&J.state[slot], (unsigned long long)sum);
    }
}

#ifndef KLMC_BAND_THREADS
#define KLMC_BAND_THREADS 1024
#endif
constexpr int kBandThreads = KLMC_BAND_THREADS;  // one CTA per SM

// Band kernel shared memory (32-bit words): rows (H + 2D) x RWb, the warps' draw
// queues, then (where they fit) K task tables of W words (rounded up to even) and
// 2 x rows words each.  A row's stride RWb is W + 5 words rounded up to 4, so that rows
// start on 16-byte boundaries and a row of the bit store (at most W + 3 words) lands
// there by one bulk copy.
__host__ __device__ __forceinline__ int band_row_words(int W)
{
    return (W + 5 + 3) / 4 * 4;
}

__host__ __device__ __forceinline__ int band_table_rows(int H, int K)
{
    return (H + 4 * K) / 2 + 2;  // anchor rows of a phase over H + 2(2K - 1) rows, py >= 2
}

__host__ __device__ __forceinline__ long long band_table_offset(int H, int K, int RWb)
{
    return (long long)(H + 2 * (2 * K + 1)) * RWb + (long long)kBandThreads / 32 * kDrawQueue2Words;
}

// Waits for phase `parity` of the mbarrier at shared address mbar, giving up after
// `limit` polls.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity, int limit)
{
    for (int i = 0; i < limit; ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done) : "r"(mbar), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}

constexpr int kCopyWaitPolls = 1 << 20;
constexpr int kCopyWaitPollsShort = 1 << 12;  // under the test hook (SweepJob::copy_shortfall)

// Tiled path, blocked: bands of H rows of a lattice too large for a cluster's
// shared memory, one CTA each, K phases per launch.  A CTA loads its band and
// D = 2K + 1 halo rows per side from the store `src` as it was at the launch's
// start, advances K phases with the blocked phase code above (every flip local,
// only the band's anchors counted), and writes its band to `dst`.  Reading one
// buffer and writing the other keeps every CTA's halo at the launch's starting
// state while other CTAs finish; the launch boundary orders the blocks.
// Bit stores on 16-byte boundaries move their rows by bulk copies (the TMA unit:
// one copy per row in, one per band row out); other stores word by word.
template <int THREADS>
__global__ void __launch_bounds__(THREADS, 1)
band_phases_kernel(const SweepJob J, const void *__restrict__ src, void *__restrict__ dst, int H, int K,
                   int tables, int k, int f0)
{
    constexpr int kWarps = THREADS / 32;
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ PhaseR pp[8];
    __shared__ long long red[5][kWarps];
    __shared__ __align__(8) unsigned long long copy_bar;
    // The next launch may be scheduled now; it waits for this one before it reads.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    Geo g;
    g.Lx = J.Lx; g.Ly = J.Ly; g.W = J.W; g.RW = band_row_words(J.W); g.magicW = g.W == 1 ? 0u : (uint32_t)J.magicW; g.one = g.W == 1 ? ~0u : 0u;
    g.nlast = g.Lx - 32 * (g.W - 1);
    g.k0 = J.key0; g.k1 = J.key1;
    g.sign = J.draw_lo > J.draw_hi ? 0 : (J.draw_lo == 0 ? -1 : 1);
    g.magicInner = g.W > 3 + 1 ? 0xFFFFFFFFu / (uint32_t)(g.W - 3) + 1u : 0u;
    g.tri = J.geometry == kTRI6;
    g.C = (int)gridDim.x;
    g.rank = (int)blockIdx.x;
    g.Y0 = (int)blockIdx.x * H;
    g.Y1 = min(g.Y0 + H, g.Ly);
    g.prevY = g.prevH = g.nextY = g.nextH = 0;
    uint32_t *const lat = smem;
    g.lat_addr = smem_addr(lat);
    g.D = 2 * K + 1;
    g.base = g.Y0 - g.D < 0 ? g.Y0 - g.D + g.Ly : g.Y0 - g.D;
    const int tid = threadIdx.x;
    const int Hc = g.Y1 - g.Y0;
    const int NL = Hc + 2 * g.D;
    const int RWb = g.RW;
    const bool bulk = J.packing == kPackBit && ((((uintptr_t)src) | ((uintptr_t)dst)) & 15u) == 0u &&
                      (J.pitch & 3) == 0 && J.pitch + 4 <= RWb;
    const uint32_t row_bytes = 4u * (uint32_t)J.pitch;
    const uint32_t bar = smem_addr(&copy_bar);
    if (bulk && tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    // The block's schedule and task tables need nothing of the launches before it but the
    // sweep index, which no launch of a series writes (the first launch of a series follows
    // its writers in full): a CTA whose SM is free prepares them while the previous launch's
    // last CTAs run.  The tables follow the rows and the draw queues.
    const long long s = __ldcg(&J.state[kSweepBase]) + k;
    const uint32_t s_lo = (uint32_t)(unsigned long long)s;
    const uint32_t s_hi = (uint32_t)((unsigned long long)s >> 32);
    if (tid < K) phase_table(g, K, s, f0 + tid, &pp[tid]);
    __syncthreads();
    const int tab_rows = band_table_rows(H, K);
    const int tab_w = (g.W + 1) & ~1;  // even, so that the int2 row entries stay aligned
    uint32_t *const tab_base = smem + band_table_offset(H, K, RWb);
    if (tables) {
        for (int q = 0; q < K; ++q) {
            const PhaseR P = pp[q];
            uint32_t *const t = tab_base + (size_t)q * (tab_w + 2 * tab_rows);
            const TaskTab T = {t, (int2 *)(t + tab_w), g.W, tab_rows};
            if (table_fits(g, P, T)) build_task_table<true>(P, g, T, tid, THREADS);
        }
    }
    // the warps' draw queues follow the rows (H + 2D rows of the tallest band)
    uint32_t *const dq = smem + (size_t)(H + 2 * g.D) * RWb + (size_t)(tid >> 5) * kDrawQueue2Words;
    dq[kDrawQueue2Acc + (tid & 31)] = 0u;  // the queue's accept words start at zero
    dq[kDrawQueue2Acc + 32 + (tid & 31)] = 0u;
    // Everything below reads what earlier launches on the stream wrote.
    asm volatile("griddepcontrol.wait;" ::: "memory");

    if (bulk) {
        // One bulk copy per row (pitch words, 16-byte aligned at both ends), completing
        // on one mbarrier whose expected byte count is exactly theirs.  Under the test
        // hook no copy is issued and the barrier expects the hook's bytes instead, which
        // nothing delivers: the wait runs out with no copy in flight.
        __syncthreads();
        const bool hook = J.copy_shortfall != 0;
        if (tid < 32) {
            if (tid == 0) {
                unsigned long long st;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 %0, [%1], %2;"
                             : "=l"(st)
                             : "r"(bar), "r"(hook ? (uint32_t)J.copy_shortfall : row_bytes * (uint32_t)NL)
                             : "memory");
            }
            __syncwarp();
            for (int lr = tid; !hook && lr < NL; lr += 32) {
                int y = g.Y0 - g.D + lr;
                if (y < 0) y += g.Ly;
                if (y >= g.Ly) y -= g.Ly;
                const char *from = (const char *)src + (size_t)y * row_bytes;
                const uint32_t to = smem_addr(lat + (size_t)lr * RWb);
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                    ::"r"(to), "l"(from), "r"(row_bytes), "r"(bar) : "memory");
            }
        }
        const int polls = hook ? kCopyWaitPollsShort : kCopyWaitPolls;
        const bool ok = mbar_wait(bar, 0u, polls);
        if (__syncthreads_or(!ok)) {
            // Give up on this launch: report it and leave the band unwritten.  Only a
            // copy that has not landed after the first bound can still be in flight
            // here (never under the hook); wait a second bound for it.
            if (tid == 0) atomicExch((unsigned long long *)&J.state[kFault], 1ull);
            mbar_wait(bar, 0u, polls);
            return;
        }
    } else {
        for (int idx = tid; idx < NL * g.W; idx += THREADS) {
            const int lr = idx / g.W, w = idx - lr * g.W;
            int y = g.Y0 - g.D + lr;
            if (y < 0) y += g.Ly;
            if (y >= g.Ly) y -= g.Ly;
            lat[(size_t)lr * RWb + w] = store_word(src, J.packing, J.pitch, y, w, g.Lx);
        }
    }
    __syncthreads();

    Acc A = {0u, 0u, 0u, 0};
    const DrawThr DT = draw_thresholds(J);
    for (int j = 0; j < K; ++j) {
        const PhaseR P = pp[j];
        uint32_t *const t = tab_base + (size_t)j * (tab_w + 2 * tab_rows);
        const TaskTab T = {t, (int2 *)(t + tab_w), g.W, tab_rows};
        const TaskTab *const tt = tables ? &T : nullptr;
        if (J.geometry == kTRI6) {
            if (g.W >= kInnerRowWords) run_phase_pair_oi<kTRI6, THREADS, true>(lat, g, P, DT, f0 + j, s_lo, s_hi, A, dq, tt, J.rk);
            else run_phase_pair_oi<kTRI6, THREADS, false>(lat, g, P, DT, f0 + j, s_lo, s_hi, A, dq, tt, J.rk);
        } else {
            if (g.W >= kInnerRowWords) run_phase_pair_oi<kSQ4, THREADS, true>(lat, g, P, DT, f0 + j, s_lo, s_hi, A, dq, tt, J.rk);
            else run_phase_pair_oi<kSQ4, THREADS, false>(lat, g, P, DT, f0 + j, s_lo, s_hi, A, dq, tt, J.rk);
        }
        __syncthreads();
    }

    if (bulk) {
        // One bulk copy per row: flips left the words and bits past its end as they were read.
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid < 32) {
            for (int r = tid; r < Hc; r += 32) {
                char *to = (char *)dst + (size_t)(g.Y0 + r) * row_bytes;
                const uint32_t from = smem_addr(lat + (size_t)(r + g.D) * RWb);
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                             ::"l"(to), "r"(from), "r"(row_bytes) : "memory");
            }
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
    } else {
        for (int idx = tid; idx < Hc * g.W; idx += THREADS) {
            const int r = idx / g.W, w = idx - r * g.W;
            const int y = g.Y0 + r;
            write_word(dst, J.packing, J.pitch, y, w, g.Lx, lat[(size_t)(r + g.D) * RWb + w]);
        }
    }

    long long att = 0;
    if (blockIdx.x == 0 && tid == 0)
        for (int j = 0; j < K; ++j) att += pp[j].att;  // the whole lattice's, counted once
    long long vals[5] = {att, (long long)A.unl, (long long)A.drw, (long long)A.acc,
                         2ll * A.dn};
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const long long ws = warp_sum(vals[q]);
        if ((tid & 31) == 0) red[q][tid >> 5] = ws;
    }
    __syncthreads();
    if (tid < 5) {
        long long sum = 0;
        for (int w = 0; w < kWarps; ++w) sum += red[tid][w];
        if (sum != 0) {
            const int slot = tid == 4 ? kNUnlike : kAttempts + tid;
            atomicAdd((unsigned long long *)&J.state[slot], (unsigned long long)sum);
        }
    }
    // The rows' copies have left shared memory (they complete with the launch).
    if (bulk && tid < 32) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

// Three variants: 512 threads (one CTA per SM; phases of many words), 256 threads with
// at most 128 registers (two CTAs per SM), of both the last warp without tasks, and 128
// threads with at most 128 registers (four CTAs per SM; batches of many lattices).
template <int THREADS, int MINB>
cudaError_t configure_once()
{
    static thread_local int configured_device = -1;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (configured_device == dev) return cudaSuccess;
    e = cudaFuncSetAttribute(resident_sweep_kernel<THREADS, MINB>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, resident_max_smem_bytes());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(resident_sweep_kernel<THREADS, MINB>,
                                 cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) configured_device = dev;
    return e;
}

cudaError_t launch(const SweepJob *d_jobs, const SweepCall *d_calls, const int *d_map,
                   const SweepJob &job0, const SweepCall &call0, int n_jobs, int cluster,
                   int threads, size_t smem_bytes, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(n_jobs * cluster), 1, 1);
    cfg.dynamicSmemBytes = smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e;
    if (threads == 512) {
        e = configure_once<512, 1>();
        if (e != cudaSuccess) return e;
        cfg.blockDim = dim3(512, 1, 1);
        e = cudaLaunchKernelEx(&cfg, resident_sweep_kernel<512, 1>, d_jobs, d_calls, d_map, job0, call0);
    } else if (threads == 128) {
        e = configure_once<128, 4>();
        if (e != cudaSuccess) return e;
        cfg.blockDim = dim3(128, 1, 1);
        e = cudaLaunchKernelEx(&cfg, resident_sweep_kernel<128, 4>, d_jobs, d_calls, d_map, job0, call0);
    } else {
        e = configure_once<256, 2>();
        if (e != cudaSuccess) return e;
        cfg.blockDim = dim3(256, 1, 1);
        e = cudaLaunchKernelEx(&cfg, resident_sweep_kernel<256, 2>, d_jobs, d_calls, d_map, job0, call0);
    }
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace

size_t resident_smem_bytes(int Lx, int Ly, int cluster)
{
    const size_t RW = (size_t)(Lx + 95) / 32;  // ceil(Lx / 32) + 2
    const int C = cluster < 1 ? 1 : cluster;
    const size_t H = (size_t)((Ly + C - 1) / C);  // tallest band
    const int K = block_phases(Lx, Ly, C);
    if (K > 1) return RW * (H + 6 * (size_t)(2 * K + 1)) * sizeof(uint32_t);  // rows + mailboxes
    return RW * (H + 4) * sizeof(uint32_t);
}

size_t resident_launch_bytes(int Lx, int Ly, int cluster)
{
    const int C = cluster < 1 ? 1 : cluster;
    const int K = block_phases(Lx, Ly, C), hmax = (Ly + C - 1) / C, W = (Lx + 31) / 32;
    const size_t rows = resident_smem_bytes(Lx, Ly, C);
    const size_t all = (size_t)(4 * (resident_row_words(W + 2, hmax, K) + chunk_table_words(W, hmax, K)));
    return all <= (size_t)kResidentMaxSmem ? all : rows;
}

int resident_max_smem_bytes() { return kResidentMaxSmem; }

int resident_block_phases(int Lx, int Ly, int cluster) { return block_phases(Lx, Ly, cluster); }

// A phase of a lattice spread over a cluster lasts as long as its busiest warp, so the
// CTA has enough threads for one task each: 224 of 256 or 480 of 512 run tasks (the
// others prepare).  GB300, us per phase at 256 / 512 threads: 64^2 on 2 CTAs 0.77 /
// 0.80, 280^2 on 16 0.91 / 0.93, 330^2 on 16 (198 words a phase) 1.01 / 1.01, 262^2 on
// 8 (216) 1.01 / 1.04, 400^2 on 16 (260) 1.21 / 1.09.
int resident_default_threads(int Lx, int Ly, int cluster)
{
    const int C = cluster < 1 ? 1 : cluster, K = block_phases(Lx, Ly, C);
    const int rows = (Ly + C - 1) / C + (K > 1 ? 2 * (2 * K - 1) : 0);
    return (long long)((rows + 1) / 2) * ((Lx + 31) / 32) > 224 ? 512 : 256;
}

int resident_max_cluster(int Ly)
{
    int c = 16;
    while (c > 1 && Ly / c < 4) c >>= 1;
    return c;
}

cudaError_t launch_resident_sweep(const SweepJob *d_jobs, const SweepCall *d_calls,
                                  const int *d_map, int n_jobs, int cluster, int threads,
                                  size_t smem_bytes, cudaStream_t stream)
{
    if (n_jobs <= 0) return cudaSuccess;
    SweepJob none_job;
    SweepCall none_call;
    memset(&none_job, 0, sizeof(none_job));
    memset(&none_call, 0, sizeof(none_call));
    return launch(d_jobs, d_calls, d_map, none_job, none_call, n_jobs, cluster, threads, smem_bytes,
                  stream);
}

cudaError_t launch_resident_sweep_one(const SweepJob &job, const SweepCall &call, int cluster,
                                      int threads, size_t smem_bytes, cudaStream_t stream)
{
    return launch(nullptr, nullptr, nullptr, job, call, 1, cluster, threads, smem_bytes, stream);
}

#ifndef KLMC_TILED_BLOCK
#define KLMC_TILED_BLOCK 4
#endif

// Lattices that the automatic choice takes to the tiled path.
constexpr long long kWideBlockSites = 786432;

TiledPlan tiled_band_plan(int Lx, int Ly, int sm_count)
{
    TiledPlan p;
    const int RWb = band_row_words((Lx + 31) / 32);
    const long long W = (((Lx + 31) / 32) + 1) & ~1ll;
    // Blocks of 8 phases halve the launches, of which each takes 5 us beside its phases; their
    // wider halos cost nothing while a phase's words, with the halo's, are one per thread
    // (1447 x 1021 square: 3.3 -> 3.0 us per phase; 8192^2 would lose 5%).
    const long long Hs = (Ly + sm_count - 1) / sm_count;
    const bool wide = (long long)Lx * Ly >= kWideBlockSites && (Hs + 2 * 15 + 1) / 2 * ((Lx + 31) / 32) <= kBandThreads;
    for (int K = wide ? 8 : KLMC_TILED_BLOCK; K >= 2; K >>= 1) {
        const int D = 2 * K + 1;
        long long H = (Ly + sm_count - 1) / sm_count;  // one CTA per SM
        // rows and draw queues must fit: shrink the bands (more bands than SMs)
        // until they do
        while (H >= 1 && 4 * band_table_offset((int)H, K, RWb) > kResidentMaxSmem) --H;
        if (H < 1 || H + 2 * D > Ly) continue;  // a band's rows must not wrap onto themselves
        const long long rows = 4 * band_table_offset((int)H, K, RWb);
        const long long tabs = 4 * K * (W + 2 * band_table_rows((int)H, K));
        p.H = (int)H;
        p.K = K;
        p.threads = kBandThreads;
        p.tables = rows + tabs <= kResidentMaxSmem ? 1 : 0;  // the task tables where they fit
        p.smem = (size_t)(rows + (p.tables ? tabs : 0));
        return p;
    }
    p.H = 0;
    p.K = 1;
    p.threads = 0;
    p.tables = 0;
    p.smem = 0;
    return p;
}

cudaError_t configure_band()
{
    static thread_local int configured_device = -1;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (configured_device == dev) return cudaSuccess;
    e = cudaFuncSetAttribute(band_phases_kernel<kBandThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kResidentMaxSmem);
    if (e == cudaSuccess) configured_device = dev;
    return e;
}

cudaError_t launch_band_phases(const SweepJob &job, const TiledPlan &plan, const void *src, void *dst,
                               int k, int f0, bool first, cudaStream_t stream)
{
    // Programmatic dependent launch: the CTAs of this launch may be scheduled while
    // the previous one drains, and wait for it in the kernel before reading.  The first of a
    // series waits for whatever is before it, as any launch.
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((job.Ly + plan.H - 1) / plan.H), 1, 1);
    cfg.blockDim = dim3(kBandThreads, 1, 1);
    cfg.dynamicSmemBytes = plan.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = first ? 0 : 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, band_phases_kernel<kBandThreads>, job, src, dst, plan.H, plan.K,
                                       plan.tables, k, f0);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace klmc
