// sweep_common.cuh -- device code shared by the resident and the tiled sweep
// kernels: the phase schedule, the anchor masks, the bit-sliced evaluation of one
// 32-site word and its draws (Philox4x32-10 from philox.cuh, which the including
// file includes at file scope).  Included inside namespace klmc.
#pragma once

struct PhaseP {
    int oi, rx, ry, px, py, umax;
    int a1, n1, a2, n2, M1;  // this band's anchor rows: m in [a1, a1+n1) u [a2, a2+n2)
    int ntask;
    int att;  // attempts of the phase over the whole lattice
};

// floor(a / 2^sh) and ceil(a / 2^sh) for any sign of a (the row spacing py of an
// anchor sublattice is 2 or 4, so every division of the schedule is a shift).
__device__ __forceinline__ int floor_shr(int a, int sh) { return a >> sh; }
__device__ __forceinline__ int ceil_shr(int a, int sh) { return -((-a) >> sh); }

// Phase parameters of (sweep s, phase f) and this band's share of its anchor rows.
// Orientation 1 is (0,1) in both geometries.
__device__ void phase_params(int geometry, int Lx, int Ly, int W, int Y0, int Y1, uint32_t k0,
                             uint32_t k1, long long s, int f, PhaseP *P)
{
    Philox4 w = philox4(0xFFFFFFFFu, (uint32_t)f, (uint32_t)(unsigned long long)s,
                        (uint32_t)((unsigned long long)s >> 32), k0, k1);
    const int nO = geometry == kTRI6 ? 3 : 2;
    const int oi = (int)__umulhi(w.v[0], (uint32_t)nO);
    const int rx = (int)__umulhi(w.v[1], (uint32_t)Lx);
    const int ry = (int)__umulhi(w.v[2], (uint32_t)Ly);
    int px, py, Kx, My;
    if (oi == 1) {
        px = 2; py = 4;
        Kx = (Lx - 2) / 2 + 1;
        My = (Ly - 3) / 4 + 1;
    } else {
        px = 4; py = 2;
        Kx = (Lx - 3) / 4 + 1;
        My = (Ly - 2) / 2 + 1;
    }
    // Anchor rows y_m = (ry + py m) mod Ly, m < My: unwrapped for m < M1.
    const int sh = py == 4 ? 2 : 1;
    const int M1 = min(My, ceil_shr(Ly - ry, sh));
    const int a1 = max(ceil_shr(Y0 - ry, sh), 0);
    const int b1 = min(floor_shr(Y1 - 1 - ry, sh), M1 - 1);
    const int a2 = max(ceil_shr(Y0 + Ly - ry, sh), M1);
    const int b2 = min(floor_shr(Y1 - 1 + Ly - ry, sh), My - 1);
    P->oi = oi; P->rx = rx; P->ry = ry; P->px = px; P->py = py;
    P->umax = px * (Kx - 1);
    P->a1 = a1; P->n1 = max(0, b1 - a1 + 1);
    P->a2 = a2; P->n2 = max(0, b2 - a2 + 1);
    P->M1 = M1;
    P->ntask = (P->n1 + P->n2) * W;
    P->att = Kx * My;
}

// Phase parameters of (sweep s, phase f) and the anchor rows whose row lies in
// [lo, hi) modulo Ly (hi - lo <= Ly; lo may be negative and hi may exceed Ly).
// The anchor rows y_m = (ry + py m) mod Ly, m < My, come as up to four runs of
// consecutive m; task row mi (0 <= mi < c[3]) has m = a[i] + mi for the first run
// i with mi < c[i].
struct PhaseR {
    int oi, rx, ry, px, py, umax;
    int a[4], c[4];
    int ntask;
    int att;  // attempts of the phase over the whole lattice
};

__device__ void phase_ranges(int geometry, int Lx, int Ly, int W, int lo, int hi, uint32_t k0,
                             uint32_t k1, long long s, int f, PhaseR *P)
{
    Philox4 w = philox4(0xFFFFFFFFu, (uint32_t)f, (uint32_t)(unsigned long long)s,
                        (uint32_t)((unsigned long long)s >> 32), k0, k1);
    const int nO = geometry == kTRI6 ? 3 : 2;
    const int oi = (int)__umulhi(w.v[0], (uint32_t)nO);
    const int rx = (int)__umulhi(w.v[1], (uint32_t)Lx);
    const int ry = (int)__umulhi(w.v[2], (uint32_t)Ly);
    int px, py, Kx, My;
    if (oi == 1) {
        px = 2; py = 4;
        Kx = (Lx - 2) / 2 + 1;
        My = (Ly - 3) / 4 + 1;
    } else {
        px = 4; py = 2;
        Kx = (Lx - 3) / 4 + 1;
        My = (Ly - 2) / 2 + 1;
    }
    const int sh = py == 4 ? 2 : 1;
    const int M1 = min(My, ceil_shr(Ly - ry, sh));  // m < M1: y_m = ry + py m (no wrap)
    // [lo, hi) as at most two intervals of [0, Ly)
    int u[2], v[2];
    if (lo < 0) {
        u[0] = lo + Ly; v[0] = Ly; u[1] = 0; v[1] = hi;
    } else if (hi > Ly) {
        u[0] = lo; v[0] = Ly; u[1] = 0; v[1] = hi - Ly;
    } else {
        u[0] = lo; v[0] = hi; u[1] = 0; v[1] = 0;
    }
    int total = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
#pragma unroll
        for (int wr = 0; wr < 2; ++wr) {
            const int off = wr ? Ly : 0;
            int a = ceil_shr(u[q] + off - ry, sh);
            int b = floor_shr(v[q] - 1 + off - ry, sh);
            a = max(a, wr ? M1 : 0);
            b = min(b, wr ? My - 1 : M1 - 1);
            const int n = u[q] < v[q] ? max(0, b - a + 1) : 0;
            P->a[2 * q + wr] = a - total;
            total += n;
            P->c[2 * q + wr] = total;
        }
    }
    P->oi = oi; P->rx = rx; P->ry = ry; P->px = px; P->py = py;
    P->umax = px * (Kx - 1);
    P->ntask = total * W;
    P->att = Kx * My;
}

// Bits p of the word at x0 with x0 + p in [lo, hi].
__device__ __forceinline__ uint32_t range_mask(int lo, int hi, int x0)
{
    int a = max(lo - x0, 0), b = min(hi - x0, 31);
    if (a > b) return 0u;
    return (0xFFFFFFFFu >> (31 - b)) & (0xFFFFFFFFu << a);
}

// Anchors of the phase in the word at x0: x = (rx + px k) mod Lx, k < Kx.
template <typename PP>
__device__ __forceinline__ uint32_t anchor_mask(int x0, const PP &P, int Lx)
{
    const uint32_t rep = P.px == 4 ? 0x11111111u : 0x55555555u;
    const int pm = P.px - 1;
    const int hi1 = min(P.rx + P.umax, Lx - 1);
    if (x0 >= P.rx && x0 + 31 <= hi1) return rep << ((P.rx - x0) & pm);  // whole word in range
    uint32_t m = (rep << ((P.rx - x0) & pm)) & range_mask(P.rx, hi1, x0);
    const int hi2 = min(P.rx - 1, P.rx + P.umax - Lx);  // wrapped part of the anchor row
    if (hi2 >= 0) m |= (rep << ((P.rx - Lx - x0) & pm)) & range_mask(0, hi2, x0);
    return m;
}

__device__ __forceinline__ uint32_t fsr(uint32_t lo, uint32_t hi, int s)
{
    return __funnelshift_r(lo, hi, s);
}

// Full adder on bit planes.
__device__ __forceinline__ void fa(uint32_t a, uint32_t b, uint32_t c, uint32_t &s, uint32_t &cy)
{
    s = a ^ b ^ c;
    cy = (a & b) | (c & (a ^ b));
}

// Bit planes of S, the number of like neighbours an unlike pair has among the six
// sites that only one of the two touches: like a among a's three, like b among b's
// three (0..6).
struct Planes {
    uint32_t s0, s1, s2;
};

// Planes of S for unlike pairs from the exclusive neighbours u1..u3 of a and w1..w3
// of b.  With tb = ~ta, the count of u equal to ta is the 2-bit sum of the u, its
// bits complemented where ta = 0 (3 - n is the complement of n), and the count of w
// equal to tb that of the w, complemented where ta = 1; the low bit of their sum no
// longer depends on ta.  Meaningless at positions of like pairs, which no caller reads.
__device__ __forceinline__ Planes count_unlike(uint32_t ta, uint32_t u1, uint32_t u2, uint32_t u3, uint32_t w1,
                                               uint32_t w2, uint32_t w3)
{
    uint32_t su, cu, sw, cw;
    fa(u1, u2, u3, su, cu);
    fa(w1, w2, w3, sw, cw);
    const uint32_t carry = ~(su ^ ta) & (sw ^ ta);
    Planes P;
    P.s0 = ~(su ^ sw);
    P.s1 = ~(cu ^ cw) ^ carry;
    const uint32_t x = ~(cu ^ ta), y = cw ^ ta;
    P.s2 = (x & y) | (carry & (x | y));
    return P;
}

// Positions that need a draw: the exchange changes n_unlike by 2 (S - 3), so it
// raises the energy when omega > 0 and S > 3 (sign > 0), or omega < 0 and S < 3.
__device__ __forceinline__ uint32_t draw_positions(const Planes &S, int sign)
{
    return sign > 0 ? S.s2 : (sign < 0 ? ~(S.s2 | (S.s1 & S.s0)) : 0u);
}

// Acceptance of draws.  A pair with a draw has S in 4..6 (omega > 0) or 0..2
// (omega < 0), so the two low bits of S name its threshold: three registers and two
// selects per draw.  Classes whose threshold is 0 never accept (DrawThr::never).
struct DrawThr {
    uint32_t t[3];
    uint32_t never;
};

__device__ __forceinline__ DrawThr draw_thresholds(const SweepJob &J)
{
    return {{J.draw_t[0], J.draw_t[1], J.draw_t[2]}, J.draw_never};
}

// Positions whose class never accepts.  Computed beside the draws and applied to their
// results: a branch around this rare case, or a mask before the draws, lengthened every phase.
__device__ __forceinline__ uint32_t never_accepted(uint32_t s0, uint32_t s1, uint32_t never)
{
    return (~(s0 | s1) & (0u - (never & 1u))) | (s0 & (0u - ((never >> 1) & 1u))) | (s1 & (0u - (never >> 2)));
}

// Whether draw r accepts the pair at the single bit b.
__device__ __forceinline__ bool accepts(uint32_t r, uint32_t s0, uint32_t s1, uint32_t b, const uint32_t (&t)[3])
{
    const uint32_t t01 = (s0 & b) != 0u ? t[1] : t[0];
    return r <= ((s1 & b) != 0u ? t[2] : t01);
}

__device__ __forceinline__ int bit_index(uint32_t b)  // of the highest bit; -1 for 0
{
    int p;
    asm("bfind.u32 %0, %1;" : "=r"(p) : "r"(b));
    return p;
}

// n_unlike change / 2 of the accepted exchanges acc (na of them).
__device__ __forceinline__ int half_dn(const Planes &S, uint32_t acc, int na)
{
    return __popc(S.s0 & acc) + 2 * __popc(S.s1 & acc) + 4 * __popc(S.s2 & acc) - 3 * na;
}

// Where the neighbours of a 32-site word lie.  A shared-memory row is W words of
// sites, the bits of its last word past the row's end zero.  l, r: distance in words
// to the word on its left and right -- around the row's ends those of the same row
// (periodic), or the last one of the row before and the first one of the row after
// (helical).  top: the bit of the left word's last site; end: the bit of the word's
// own last site.  (Rows with copies of their end sites on either side need no such
// distances, but every flip near an end then mends copies: that took 0.15-0.21 us of a
// 1.0-1.4 us phase of a 64^2 or 400^2 lattice on a cluster.)
struct WordEnds {
    int l, r;
    int top, end;
    bool fix;  // a last word of one site (Lx mod 32 = 1): this word is it or the one before,
    int fix2;  // which is then followed by the word at this distance
};

// nlast: sites of a row's last word; hrow: 0 (periodic) or the row stride (helical).
__device__ __forceinline__ WordEnds word_ends(int j, int W, int nlast, int hrow)
{
    const bool first = j == 0, last = j == W - 1;
    WordEnds E;
    E.l = first ? W - 1 - hrow : -1;
    E.r = last ? 1 - W + hrow : 1;
    E.top = first ? nlast - 1 : 31;
    E.end = last ? nlast - 1 : 31;
    E.fix = nlast == 1 && j >= W - 2;
    E.fix2 = 2 - W + hrow;
    return E;
}

// How a word's windows are taken: kPlain, the words beside it are its neighbours (one funnel
// shift per window); kEnds, it may be at an end of its row; kFix, and rows may have a last
// word of one site.
enum Windows { kPlain, kEnds, kFix };

// The sites at distance -1, +1 and +2 of the word at p (32 at a time).
template <Windows WN>
__device__ __forceinline__ uint32_t window_m1(const uint32_t *p, const WordEnds &E)
{
    if (WN == kPlain) return __funnelshift_r(p[-1], p[0], 31);
    return p[0] + p[0] + (p[E.l] >> E.top);  // bits above the left word's last site are zero
}
template <Windows WN>
__device__ __forceinline__ uint32_t window_p1(const uint32_t *p, const WordEnds &E)
{
    if (WN == kPlain) return __funnelshift_r(p[0], p[1], 1);
    return (p[0] >> 1) + p[E.r] * (1u << E.end);
}
template <Windows WN>
__device__ __forceinline__ uint32_t window_p2(const uint32_t *p, const WordEnds &E)
{
    if (WN == kPlain) return __funnelshift_r(p[0], p[1], 2);
    const uint32_t r = p[E.r];
    uint32_t v = (p[0] >> 2) + r * ((1u << E.end) >> 1);
    // (the sum's bits past the row's end carry nothing into it; with a last word of one
    // site, that word's site and the last one before it look two words on)
    if (WN == kFix && E.fix) v = E.end == 0 ? r >> 1 : (v & 0x7FFFFFFFu) | (p[E.fix2] << 31);
    return v;
}

// Bit-sliced evaluation of the word at p of an anchor row in shared memory (rows of
// stride RW): the types ta, tb of a = (x, y) and b = a + o for its 32 positions, and
// the bit planes of S.  A pair that moves is unlike, so a neighbour of both sites is
// like exactly one of them and adds a constant: only the six neighbours of one site
// alone are compared (10 comparisons and adders of 10 inputs before, 6 now).
template <int G, int OI, Windows WN>
__device__ __forceinline__ void evaluate(const uint32_t *p, int RW, const WordEnds &E, uint32_t &ta, uint32_t &tb,
                                         Planes &S)
{
    const uint32_t *pm = p - RW, *pp = p + RW;
    ta = p[0];
    const uint32_t Am = window_m1<WN>(p, E);
    if (G == kTRI6 && OI == 0) {
        // a: (-1,0) (0,-1) (-1,1); b = (1,0): (2,0) (1,1) (2,-1); common (0,1) (1,-1)
        tb = window_p1<WN>(p, E);
        S = count_unlike(ta, Am, pm[0], window_m1<WN>(pp, E), window_p2<WN>(p, E), window_p1<WN>(pp, E), window_p2<WN>(pm, E));
    } else if (G == kTRI6 && OI == 1) {
        // a: (-1,0) (0,-1) (1,-1); b = (0,1): (1,1) (0,2) (-1,2); common (1,0) (-1,1)
        const uint32_t *pq = pp + RW;
        tb = pp[0];
        S = count_unlike(ta, Am, pm[0], window_p1<WN>(pm, E), window_p1<WN>(pp, E), pq[0], window_m1<WN>(pq, E));
    } else if (G == kTRI6 && OI == 2) {
        // a: (-1,0) (0,1) (-1,1); b = (1,-1): (2,-1) (1,-2) (2,-2); common (1,0) (0,-1)
        const uint32_t *pn = pm - RW;
        tb = window_p1<WN>(pm, E);
        S = count_unlike(ta, Am, pp[0], window_m1<WN>(pp, E), window_p2<WN>(pm, E), window_p1<WN>(pn, E), window_p2<WN>(pn, E));
    } else if (G == kSQ4 && OI == 0) {
        // a: (-1,0) (0,1) (0,-1); b = (1,0): (2,0) (1,1) (1,-1)
        tb = window_p1<WN>(p, E);
        S = count_unlike(ta, Am, pp[0], pm[0], window_p2<WN>(p, E), window_p1<WN>(pp, E), window_p1<WN>(pm, E));
    } else {
        // SQ4; a: (1,0) (-1,0) (0,-1); b = (0,1): (1,1) (-1,1) (0,2)
        tb = pp[0];
        S = count_unlike(ta, window_p1<WN>(p, E), Am, pm[0], window_p1<WN>(pp, E), window_m1<WN>(pp, E), pp[RW]);
    }
}

// Partners b = a + o of the accepted anchors acc of a word with ends E: their mask in
// the word at the same place of b's row, and (returned) the one that falls into the
// word on its right, as its bit 0.
template <int OI, Windows WN = kEnds>
__device__ __forceinline__ uint32_t partners(uint32_t acc, const WordEnds &E, uint32_t &b)
{
    if (OI == 1) {
        b = acc;
        return 0u;
    }
    if (WN == kPlain) {
        b = acc << 1;
        return acc >> 31;
    }
    b = (acc << 1) & (2u * (1u << E.end) - 1u);
    return (acc >> E.end) & 1u;
}

// Accept bits of the positions in dmask, each drawing Philox word 0 of counter
// {site_base + p, f, s_lo, s_hi}; two evaluations interleaved at a time (after an odd
// last draw the second one's bit is 0).  The first two are drawn without a test for
// any: nearly every warp has a lane that needs them, and without the branch they are
// scheduled into the evaluation.  The round keys are added up in every draw: sixteen
// registers of them cost more than the additions.  (400^2 on 16 CTAs: 1.32 -> 1.18 us
// per phase; 256 uneven replicas on 128 threads per CTA: 177 -> 162 us per sweep.)
__device__ __forceinline__ uint32_t draw_accepts(uint32_t dmask, const Planes &S, uint32_t site_base,
                                                 const DrawKey &dk, const DrawThr &T)
{
    uint32_t acc = 0u;
    uint32_t dm = dmask;
    do {
        const uint32_t b1 = dm & (0u - dm);
        dm ^= b1;
        const uint32_t b2 = dm & (0u - dm);
        dm ^= b2;
        uint32_t r1, r2;
        philox2_w0_key(site_base + (uint32_t)bit_index(b1), site_base + (uint32_t)bit_index(b2), dk, r1, r2);
        if (accepts(r1, S.s0, S.s1, b1, T.t)) acc |= b1;
        if (accepts(r2, S.s0, S.s1, b2, T.t)) acc |= b2;
    } while (dm != 0u);
    return acc & ~never_accepted(S.s0, S.s1, T.never);
}

// Accept bits of two tasks per lane (t and t + THREADS) when the warp's draws are
// drawn by all its lanes.  Every lane stores each task's S planes and first site
// index once, and appends its draws (task, lane, bit) as 16-bit entries to the
// warp's queue at its prefix-sum offset; then lane i draws entries i and i + 32 of
// every 64 (two Philox chains interleaved), reading the entry's S and site from
// its record, and returns accepted bits through the warp's accept words with
// shared atomics.  One scan and one pass serve both tasks, so a pass drains about
// twice the draws of one task per lane.  When the warp has more than kDrawQueue2
// draws, each lane draws its own.  Every lane of the warp must call it.  Region q
// (16-byte aligned, kDrawQueue2Words words): records uint4[2][32] (the two low planes
// of S and the first site), accept words uint32[2][32] (zero on entry and on return),
// entries uint16[kDrawQueue2].
constexpr int kDrawQueue2 = 512;
constexpr int kDrawQueue2Acc = 2 * 32 * 4;  // word offset of the accept words
constexpr int kDrawQueue2Words = kDrawQueue2Acc + 2 * 32 + kDrawQueue2 / 2;

__device__ __forceinline__ void draw_accepts_queue2(uint32_t dmask0, const Planes &S0, uint32_t base0,
                                                    uint32_t dmask1, const Planes &S1, uint32_t base1,
                                                    const DrawKey &dk, const uint32_t (&rk)[2][8],
                                                    const DrawThr &T, uint32_t *q, uint32_t &acc0,
                                                    uint32_t &acc1)
{
    acc0 = 0u;
    acc1 = 0u;
    if (T.never != 0u) {
        dmask0 &= ~never_accepted(S0.s0, S0.s1, T.never);
        dmask1 &= ~never_accepted(S1.s0, S1.s1, T.never);
    }
    if (!__any_sync(0xFFFFFFFFu, (dmask0 | dmask1) != 0u)) return;
    const int lane = (int)(threadIdx.x & 31);
    const int nd0 = __popc(dmask0), nd = nd0 + __popc(dmask1);
    int incl = nd;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += v;
    }
    const int total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    if (total > kDrawQueue2) {
        acc0 = draw_accepts(dmask0, S0, base0, dk, T);
        acc1 = draw_accepts(dmask1, S1, base1, dk, T);
        return;
    }
    uint4 *const rec = (uint4 *)q;  // [2][32]
    uint32_t *const wacc = q + kDrawQueue2Acc;  // [2][32]
    uint16_t *const ent = (uint16_t *)(wacc + 64);
    if (dmask0 != 0u) rec[lane] = make_uint4(S0.s0, S0.s1, base0, 0u);
    if (dmask1 != 0u) rec[32 + lane] = make_uint4(S1.s0, S1.s1, base1, 0u);
    int slot = incl - nd;
    uint32_t dm = dmask0;
    while (dm != 0u) {
        const int p = __ffs(dm) - 1;
        dm &= dm - 1u;
        ent[slot++] = (uint16_t)(((uint32_t)lane << 5) | (uint32_t)p);
    }
    dm = dmask1;
    while (dm != 0u) {
        const int p = __ffs(dm) - 1;
        dm &= dm - 1u;
        ent[slot++] = (uint16_t)(1024u | ((uint32_t)lane << 5) | (uint32_t)p);
    }
    __syncwarp();
    // Rounds of 64 entries, lane i taking entries i and i + 32 (two Philox chains);
    // a last round of at most 32 entries takes one chain per lane.
    for (int k0 = 0; k0 < total; k0 += 64) {
        const int k = k0 + lane;
        if (total - k0 > 32) {
            const uint32_t e1 = ent[k];
            const bool two = k + 32 < total;
            const uint32_t e2 = two ? ent[k + 32] : e1;
            const uint32_t r1i = e1 >> 5, p1 = e1 & 31u, r2i = e2 >> 5, p2 = e2 & 31u;  // record = task*32 + lane
            const uint4 a = rec[r1i], b = rec[r2i];
            uint32_t r1, r2;
            philox2_w0_rk(a.z + p1, b.z + p2, dk, rk, r1, r2);
            if (accepts(r1, a.x, a.y, 1u << p1, T.t)) atomicOr(wacc + r1i, 1u << p1);
            if (two && accepts(r2, b.x, b.y, 1u << p2, T.t)) atomicOr(wacc + r2i, 1u << p2);
        } else if (k < total) {
            const uint32_t e1 = ent[k];
            const uint32_t r1i = e1 >> 5, p1 = e1 & 31u;
            const uint4 a = rec[r1i];
            const uint32_t r1 = philox_w0_rk(a.z + p1, dk, rk);
            if (accepts(r1, a.x, a.y, 1u << p1, T.t)) atomicOr(wacc + r1i, 1u << p1);
        }
    }
    __syncwarp();
    acc0 = wacc[lane];
    acc1 = wacc[32 + lane];
    wacc[lane] = 0u;
    wacc[32 + lane] = 0u;
    __syncwarp();
}

// Word w (32 sites) of row y of the device store, the bits past the row's end zero.
__device__ __forceinline__ uint32_t store_word(const void *lat, int packing, int pitch, int y, int w,
                                               int Lx)
{
    const int n = min(32, Lx - 32 * w);
    if (packing == kPackBit) {
        const uint32_t v = ((const uint32_t *)lat)[(size_t)y * pitch + w];
        return n < 32 ? v & ((1u << n) - 1u) : v;
    }
    // rows of a multiple of 16 bytes, zeros past the last site: four sites at a time
    const uint8_t *const bytes = (const uint8_t *)lat + (size_t)y * pitch + 32 * w;
    const uint32_t *const row = (const uint32_t *)bytes;
    uint32_t v = 0u;
    if ((uintptr_t)bytes & 3u) {  // a caller's allocator
        for (int b = 0; b < n; ++b) v |= (uint32_t)(bytes[b] & 1u) << b;
        return v;
    }
    for (int q = 0; 4 * q < n; ++q) {
        const uint32_t b = row[q];  // bytes of 0 or 1
        v |= ((b & 1u) | ((b >> 7) & 2u) | ((b >> 14) & 4u) | ((b >> 21) & 8u)) << (4 * q);
    }
    return n < 32 ? v & ((1u << n) - 1u) : v;
}

// Writes word w of row y to the device store (sites only).
__device__ __forceinline__ void write_word(void *lat, int packing, int pitch, int y, int w, int Lx, uint32_t v)
{
    if (packing == kPackBit) {
        ((uint32_t *)lat)[(size_t)y * pitch + w] = v;
        return;
    }
    const int n = min(32, Lx - 32 * w);
    uint8_t *const bytes = (uint8_t *)lat + (size_t)y * pitch + 32 * w;
    uint32_t *const row = (uint32_t *)bytes;
    if ((uintptr_t)bytes & 3u) {  // a caller's allocator
        for (int b = 0; b < n; ++b) bytes[b] = (uint8_t)((v >> b) & 1u);
        return;
    }
    for (int q = 0; 4 * q < n; ++q) {
        const uint32_t b = v >> (4 * q);
        row[q] = (b & 1u) | ((b & 2u) << 7) | ((b & 4u) << 14) | ((b & 8u) << 21);
    }
}
