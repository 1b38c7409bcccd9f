// sweep_helical.cu -- Kawasaki exchange sweeps of the helical triangular lattice
// with the seven-colour schedule of the paper's MPKK loop (section "Massive
// Parallel Kawasaki Kinetics", Fig. 4), the lattice resident in the shared memory
// of a thread-block cluster for the whole launch and evaluated 32 sites per thread.
//
// Helical boundary: site i's neighbours are (i + d) mod N for the six axial steps
// d = dx + dy*Lx.  Read row by row, position p of row y is site (y*Lx + p) mod N:
// position -1 is the last site of row y-1 and positions Lx, Lx+1 are the first two
// sites of row y+1.  So the bit-sliced evaluation of the periodic kernels applies
// with the windows of a row's end words reaching into the rows beside it (WordEnds).
//
// Iteration f of sweep s draws the coverage k and one direction d from Philox at
// {0xFFFFFFFF, f, s_lo, s_hi}; every centre c (c mod 7 = k) attempts the
// exchange with c + D[d].  Direction d is orientation o = d/2 of (1,0), (0,1),
// (1,-1), forward for even d and backward for odd d; a backward pair {c - o, c}
// is evaluated as the forward pair of its anchor a = c - o, whose residue mod 7 is
// k - step(o).  So every iteration is one orientation and one residue class of
// anchors, 4 to 5 per 32-site word in every row, and the draw of anchor a uses
// the counter of its centre, {c, f, s_lo, s_hi}.
//
// Work split as in the periodic resident kernel: CTA r of a C-CTA cluster owns
// rows [Y_r, Y_r+1) and holds D = 2K + 1 halo rows per side; it advances K
// iterations alone, evaluating in the j-th of them the anchors within
// 2 (K - 1 - j) + 1 rows of its band (a pair's evaluation and its flips reach two
// rows, the windows around row ends included), and only anchors of its own band are
// counted.  Then the halo exchange of cluster_exchange.cuh.  Iterations run across
// sweep boundaries (seven per sweep).  A thread's first word is the same in every
// iteration, so its place and ends are found once; the next iteration's schedule entry
// and draw key are prepared by one lane.  Bound: the instructions of an iteration's
// busiest warp (402 x 399 on 16 CTAs: 1.24 us per iteration; 1.88 with copies of the row
// ends and a cluster barrier per exchange).
#include <string.h>

#include "klmc_internal.h"
#include "philox.cuh"

namespace klmc {
namespace {

#include "sweep_common.cuh"
#include "cluster_exchange.cuh"

constexpr int kHelicalThreads = 512;
constexpr int kHelicalMaxSmem = 227 * 1024 - 6144;

__device__ __forceinline__ void hred_xor(uint32_t addr, uint32_t v)
{
    asm volatile("red.shared.xor.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ uint32_t hcluster_nctarank()
{
    uint32_t v;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(v));
    return v;
}

__device__ __forceinline__ uint32_t hcluster_ctarank()
{
    uint32_t v;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(v));
    return v;
}

template <typename T>
__device__ __forceinline__ T hwarp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// Iterations per block for Lx x Ly over C CTAs: the largest K of 4, 2 whose halo
// D = 2K + 1 fits every band (twice for C = 2) and whose rows and mailboxes fit in
// shared memory; 0 when none does (the per-iteration kernel runs the lattice).
__host__ __device__ __forceinline__ int helical_block(int Lx, int Ly, int C)
{
    if (C < 2) return 0;
    const int hmin = Ly / C, hmax = (Ly + C - 1) / C;
    const long long RW = (Lx + 95) / 32;
    for (int K = 4; K >= 2; K >>= 1) {
        const int D = 2 * K + 1;
        if (D > hmin || (C == 2 && 2 * D > hmin)) continue;
        if (RW * (hmax + 6 * D) * 4 > kHelicalMaxSmem) continue;
        return K;
    }
    return 0;
}

struct HGeo {
    int Lx, Ly, W, RW, D, H, Y0, C, rank, sign, NL, nlast;
    long long N;
    uint32_t k0, k1, lat_addr;
};

// An iteration's schedule entry, prepared one iteration ahead by one lane.
struct __align__(16) HSched {
    int oi, kr;       // orientation, anchors' residue mod 7
    int delta;        // from an anchor to its centre's site
    uint32_t hk, la;  // the iteration's part of the draw key
};

// A thread's word of an iteration, relative to the iteration's first row; the same in every
// iteration.
struct HWord {
    int row, j;
    WordEnds E;
};

struct HAcc {
    uint32_t unl, drw, acc;
    int32_t dn;
};

// Accept bits of the positions in dmask; the draw of position p uses the counter
// of site (base + p) mod N.  32-bit arithmetic: a lattice resident in one
// cluster's shared memory has far fewer than 2^30 sites, and base lies within
// [-Lx, N + Lx).
__device__ __forceinline__ uint32_t helical_draws(uint32_t dmask, const Planes &S, int base, int N,
                                                  const DrawKey &dk, const DrawThr &T)
{
    uint32_t acc = 0u;
    uint32_t dm = dmask;
    do {
        const uint32_t b1 = dm & (0u - dm);
        dm ^= b1;
        const uint32_t b2 = dm & (0u - dm);  // 0 after an odd last draw
        dm ^= b2;
        int c1 = base + bit_index(b1), c2 = base + bit_index(b2);
        c1 += c1 >= N ? -N : (c1 < 0 ? N : 0);
        c2 += c2 >= N ? -N : (c2 < 0 ? N : 0);
        uint32_t r1, r2;
        philox2_w0_key((uint32_t)c1, (uint32_t)c2, dk, r1, r2);
        if (accepts(r1, S.s0, S.s1, b1, T.t)) acc |= b1;
        if (accepts(r2, S.s0, S.s1, b2, T.t)) acc |= b2;
    } while (dm != 0u);
    return acc & ~never_accepted(S.s0, S.s1, T.never);
}

__device__ __forceinline__ HWord helical_word(const HGeo &g, int t)
{
    HWord w;
    w.row = t / g.W;
    w.j = t - w.row * g.W;
    w.E = word_ends(w.j, g.W, g.nlast, g.RW);
    return w;
}

// One iteration: anchors of the entry's residue in local rows [lr0, lr0 + nrows),
// orientation OI, draw counters shifted to the centres.  w: the thread's first word.
template <int OI, Windows WN>
__device__ __forceinline__ void helical_iteration(const uint32_t *lat, const HGeo &g, const HSched &c, int lr0, int nrows,
                                                  HWord w, const DrawKey &dk, const DrawThr &T, HAcc &A)
{
    // b = a + o: (1,0) -> same row, +1; (0,1) -> next row; (1,-1) -> previous row, +1
    const uint32_t rowbytes = 4u * (uint32_t)g.RW;
    const int ntask = nrows * g.W;
    for (int t = (int)threadIdx.x; t < ntask;) {
        const int lr = lr0 + w.row;
        int y = g.Y0 - g.D + lr;
        y = y < 0 ? y + g.Ly : (y >= g.Ly ? y - g.Ly : y);
        const uint32_t a0 = (uint32_t)y * (uint32_t)g.Lx + 32u * (uint32_t)w.j;  // site of position 0 (< N < 2^31)
        // anchors: positions p with (a0 + p) = kr mod 7, below Lx
        int o = c.kr - (int)(a0 % 7u);
        o += o < 0 ? 7 : 0;
        // bits o, o+7, o+14, o+21, o+28; word W-1 ends at bit E.end
        const uint32_t am = (0x10204081u << o) & (2u * (1u << w.E.end) - 1u);
        uint32_t ta, tb;
        Planes S;
        const uint32_t *const p = lat + lr * g.RW + w.j;
        evaluate<kTRI6, OI, WN>(p, g.RW, w.E, ta, tb, S);
        const uint32_t unl = (ta ^ tb) & am;
        const uint32_t dmask = unl & draw_positions(S, g.sign);
        const uint32_t acc = (unl & ~dmask) | helical_draws(dmask, S, (int)a0 + c.delta, (int)g.N, dk, T);
        const uint32_t own = (unsigned)(lr - g.D) < (unsigned)g.H ? ~0u : 0u;
        const uint32_t oacc = acc & own;
        const int na = __popc(oacc);
        A.unl += __popc(unl & own);
        A.drw += __popc(dmask & own);
        A.acc += na;
        A.dn += half_dn(S, oacc, na);
        const uint32_t wa = smem_addr(p);
        const uint32_t wb = OI == 0 ? wa : (OI == 1 ? wa + rowbytes : wa - rowbytes);
        uint32_t b;
        const uint32_t next = partners<OI>(acc, w.E, b);
        if (OI == 0) {
            hred_xor(wa, acc | b);
        } else {
            hred_xor(wa, acc);
            hred_xor(wb, b);
        }
        if (OI != 1) hred_xor(wb + 4u * (uint32_t)w.E.r, next);
        t += kHelicalThreads;
        if (t < ntask) w = helical_word(g, t);
    }
}

// Iteration f of sweep s: the colour kc in [0, 7) and the direction draw d in [0, 6)
// (orientation d / 2, backward pair when d is odd), from the schedule's Philox block.
__device__ __forceinline__ void helical_sched(const HGeo &g, unsigned long long s, int f, HSched *c)
{
    const Philox4 w = philox4(0xFFFFFFFFu, (uint32_t)f, (uint32_t)s, (uint32_t)(s >> 32), g.k0, g.k1);
    const int kc = (int)__umulhi(w.v[0], 7u), d = (int)__umulhi(w.v[1], 6u), oi = d >> 1;
    const bool back = d & 1;  // a backward pair's centre is its anchor + o
    // kr = (kc - delta) mod 7, from delta mod 7 in {0, 1, Lx mod 7, 1 - Lx mod 7}
    const int lx7 = g.Lx % 7;
    int kr = kc - (back ? (oi == 0 ? 1 : (oi == 1 ? lx7 : (lx7 <= 1 ? 1 - lx7 : 8 - lx7))) : 0);
    kr += kr < 0 ? 7 : 0;
    const DrawKey dk = draw_key((uint32_t)f, (uint32_t)s, (uint32_t)(s >> 32), g.k0, g.k1);
    c->oi = oi;
    c->kr = kr;
    c->delta = back ? (oi == 0 ? 1 : (oi == 1 ? g.Lx : 1 - g.Lx)) : 0;
    c->hk = dk.hk;
    c->la = dk.la;
}

__global__ void __launch_bounds__(kHelicalThreads, 1)
helical_resident_kernel(const SweepJob J, const SweepCall Cl)
{
    constexpr int kWarps = kHelicalThreads / 32;
    extern __shared__ __align__(16) uint32_t lat[];
    __shared__ long long red[5][kWarps];
    __shared__ HSched sched[2];  // the current and the next iteration
    __shared__ __align__(8) unsigned long long xbar[kExchangeBars];
    if (Cl.n_mcs <= 0) return;

    HGeo g;
    g.Lx = J.Lx; g.Ly = J.Ly; g.W = J.W; g.RW = J.RW;
    g.k0 = J.key0; g.k1 = J.key1;
    g.N = (long long)J.Lx * J.Ly;
    g.nlast = g.Lx - 32 * (g.W - 1);
    // The host's draw range is [z, 2(z-1)] (omega > 0), [0, z-2] (omega < 0) or empty.
    g.sign = J.draw_lo > J.draw_hi ? 0 : (J.draw_lo == 0 ? -1 : 1);
    g.C = (int)hcluster_nctarank();
    g.rank = (int)hcluster_ctarank();
    g.Y0 = (int)(((long long)g.rank * g.Ly) / g.C);
    const int Y1 = (int)(((long long)(g.rank + 1) * g.Ly) / g.C);
    g.H = Y1 - g.Y0;
    const int K = helical_block(g.Lx, g.Ly, g.C);  // >= 2: the host launches only such lattices
    g.D = 2 * K + 1;
    g.NL = g.H + 2 * g.D;
    g.lat_addr = smem_addr(lat);
    const int hmax = (g.Ly + g.C - 1) / g.C;
    const int tid = threadIdx.x;

    for (int idx = tid; idx < g.NL * g.RW; idx += kHelicalThreads) {
        const int lr = idx / g.RW, w = idx - lr * g.RW;
        int y = (g.Y0 - g.D + lr) % g.Ly;
        if (y < 0) y += g.Ly;
        lat[idx] = w < g.W ? store_word(J.lat, J.packing, J.pitch, y, w, g.Lx) : 0u;
    }
    const DrawThr T = draw_thresholds(J);
    // Iteration f of sweep s draws its colour and direction from one Philox block;
    // the last warp's lane 0 draws them one iteration ahead, off the tasks' path.
    const bool sched_lane = tid == kHelicalThreads - 32;
    if (sched_lane) helical_sched(g, (unsigned long long)Cl.sweep0, 0, &sched[0]);
    exchange_init(xbar);
    cluster_barrier();  // every CTA of the cluster runs before any peer writes into it

    const long long n_unlike0 = (tid == 0 && g.rank == 0 && Cl.trace_every > 0) ? J.state[kNUnlike] : 0;
    // Every iteration attempts one exchange per seven sites (7 | N), counted by one thread.
    const unsigned long long t_att = tid == 0 && g.rank == 0 ? (unsigned long long)(g.N * Cl.n_mcs) : 0ull;
    unsigned long long t_unl = 0, t_drw = 0, t_acc = 0;
    long long t_dn = 0;
    int jb = 0, pb = 0;  // iteration within the block; buffer of the current schedule entry
    int block = 0;
    Exchange X = exchange_for<kHelicalThreads>(xbar, g.lat_addr, g.C, g.rank, g.D * g.RW, J.copy_shortfall != 0);
    const HWord word = helical_word(g, tid);
    for (long long it = 0; it < Cl.n_mcs; ++it) {
        const unsigned long long s = (unsigned long long)(Cl.sweep0 + it);
        DrawKey dk = draw_key(0u, (uint32_t)s, (uint32_t)(s >> 32), g.k0, g.k1);
        HAcc A = {0u, 0u, 0u, 0};
#pragma unroll 1
        for (int f = 0; f < 7; ++f) {
            const HSched c = sched[pb];
            const bool last = f == 6 && it + 1 == Cl.n_mcs;
            if (sched_lane && !last) helical_sched(g, f == 6 ? s + 1 : s, f == 6 ? 0 : f + 1, &sched[pb ^ 1]);
            dk.hk = c.hk;
            dk.la = c.la;
            const int e = 2 * (K - 1 - jb) + 1;
            if (g.nlast == 1) {  // rows whose last word holds one site take a longer window
                if (c.oi == 0) helical_iteration<0, kFix>(lat, g, c, g.D - e, g.H + 2 * e, word, dk, T, A);
                else if (c.oi == 1) helical_iteration<1, kFix>(lat, g, c, g.D - e, g.H + 2 * e, word, dk, T, A);
                else helical_iteration<2, kFix>(lat, g, c, g.D - e, g.H + 2 * e, word, dk, T, A);
            } else {
                if (c.oi == 0) helical_iteration<0, kEnds>(lat, g, c, g.D - e, g.H + 2 * e, word, dk, T, A);
                else if (c.oi == 1) helical_iteration<1, kEnds>(lat, g, c, g.D - e, g.H + 2 * e, word, dk, T, A);
                else helical_iteration<2, kEnds>(lat, g, c, g.D - e, g.H + 2 * e, word, dk, T, A);
            }
            __syncthreads();
            pb ^= 1;
            const bool exch = jb == K - 1;
            jb = exch ? 0 : jb + 1;
            if (exch && !last) {
                exchange_halos<kHelicalThreads>(lat, g.lat_addr, g.RW, g.H, g.D, hmax, block++, X);
                __syncthreads();
            }
        }
        t_unl += A.unl; t_drw += A.drw; t_acc += A.acc;
        t_dn += 2 * A.dn;
        if (Cl.trace_every > 0 && (it + 1) % Cl.trace_every == 0) {
            const long long ws = hwarp_sum(t_dn);
            if ((tid & 31) == 0 && ws != 0)
                atomicAdd((unsigned long long *)&Cl.trace[(it + 1) / Cl.trace_every - 1], (unsigned long long)ws);
            if (tid == 0 && g.rank == 0)
                atomicAdd((unsigned long long *)&Cl.trace[(it + 1) / Cl.trace_every - 1],
                          (unsigned long long)n_unlike0);
        }
    }

    exchange_end(X, J.copy_shortfall != 0, J.state);

    // Write the band back (sites only).
    for (int idx = tid; idx < g.H * g.W; idx += kHelicalThreads) {
        const int r = idx / g.W, w = idx - r * g.W;
        const int y = g.Y0 + r;
        write_word(J.lat, J.packing, J.pitch, y, w, g.Lx, lat[(r + g.D) * g.RW + w]);
    }

    long long vals[5] = {(long long)t_att, (long long)t_unl, (long long)t_drw, (long long)t_acc, t_dn};
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const long long ws = hwarp_sum(vals[k]);
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

}  // namespace

int helical_resident_block(int Lx, int Ly, int cluster) { return helical_block(Lx, Ly, cluster); }

size_t helical_resident_smem_bytes(int Lx, int Ly, int cluster)
{
    const size_t RW = (size_t)(Lx + 95) / 32;
    const int C = cluster < 1 ? 1 : cluster;
    const size_t H = (size_t)((Ly + C - 1) / C);
    const int K = helical_block(Lx, Ly, C);
    return RW * (H + 6 * (size_t)(2 * (K > 0 ? K : 1) + 1)) * sizeof(uint32_t);
}

cudaError_t launch_helical_resident(const SweepJob &job, const SweepCall &call, int cluster, cudaStream_t stream)
{
    static thread_local int configured_device = -1;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (configured_device != dev) {
        e = cudaFuncSetAttribute(helical_resident_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kHelicalMaxSmem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(helical_resident_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        configured_device = dev;
    }
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)cluster, 1, 1);
    cfg.blockDim = dim3(kHelicalThreads, 1, 1);
    cfg.dynamicSmemBytes = helical_resident_smem_bytes(job.Lx, job.Ly, cluster);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, helical_resident_kernel, job, call);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace klmc
