// cluster_exchange.cuh -- the halo exchange of lattices resident in a thread-block
// cluster's shared memory, between the CTAs of neighbouring bands.  Included inside
// namespace klmc by the resident sweeps, and by tests/exchange_model.cpp, which runs
// the exchange on the host over a model of the operations below.
#pragma once

#ifndef KLMC_EXCHANGE_MODEL
__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// Distance from a shared address of this CTA to the same one of CTA `rank`.
__device__ __forceinline__ uint32_t mapa_distance(uint32_t addr, int rank)
{
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(rank));
    return remote - addr;
}

// Readies the mbarrier at shared address bar for one arrival per phase.
__device__ __forceinline__ void mbar_init(uint32_t bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// The phase's one arrival; the phase completes with it and `bytes` of stores.
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes)
{
    unsigned long long st;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 %0, [%1], %2;" : "=l"(st) : "r"(bar), "r"(bytes) : "memory");
}

// Stores v at address `to` of another CTA of the cluster and counts its 4 bytes on the
// mbarrier at address `bar` there.
__device__ __forceinline__ void store_counted(uint32_t to, uint32_t v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];"
                 ::"r"(to), "r"(v), "r"(bar) : "memory");
}

// Waits for phase `parity` of the mbarrier at shared address bar, which the stores of
// another CTA of the cluster complete; false after `limit` polls.
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, int limit)
{
    for (int i = 0; i < limit; ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}
#endif

// Polls of a wait before it gives up, and under the test hook (SweepJob::copy_shortfall).
constexpr int kExchangePolls = 1 << 20;
constexpr int kExchangePollsShort = 1 << 12;

// A CTA's mbarriers: two sides (0: from the CTA above, 1: from the one below) of two
// block parities.
constexpr int kExchangeBars = 4;

// What a thread's part in its CTA's exchanges needs: the CTA's mbarriers, the distances
// from its own shared memory to its neighbours', the polls of a wait (kExchangePollsShort:
// the test hook, under which no store is sent; 0: a wait of this thread ran out, and it
// takes no further part), and the sides whose mbarriers the thread arms (bits 0 and 1).
struct Exchange {
    uint32_t bar, to_prev, to_next;
    int polls;
    uint32_t arms;
};

__device__ __forceinline__ uint32_t exchange_bar(uint32_t bar, uint32_t side, uint32_t parity)
{
    return bar + 16u * side + 8u * parity;
}

// End of a block: the D lowest and D highest band rows go to the mailboxes of parity
// block & 1 in the neighbouring CTAs, by asynchronous stores that count their bytes on
// the receiver's mbarriers; this CTA's own mailboxes then fill its halo rows.  A CTA
// waits for its two neighbours only.  The caller has a barrier of the NT threads before
// and after.
//
// Nothing but the following orders the exchanges (a warp may stall anywhere, and
// stores of one CTA may land in any order).  A neighbour sends block n + 2 after it
// has received all of this CTA's block n + 1, which this CTA sends after its barrier
// behind exchange n: by then every byte of block n has landed and been copied.  So
// two mailboxes per side are enough, and two mbarriers: on the one of a side and parity
// the bytes of block n + 2 come after the phase of block n is complete.  One mbarrier
// per side would not do: a neighbour needs nothing of this CTA's first warp to be one
// block ahead of it, and its block n + 1 would then count in the phase of block n.
// Within a phase the arrival and the stores come in any order.
//
// A thread whose wait ran out takes no further part, and the side's mbarrier is armed by
// a thread that waits on it: so no arrival meets a phase that still lacks its bytes.  The
// waits for what that thread does not send run out in turn, a CTA further with every
// block, so that a barrier left behind takes the bytes of at most as many blocks as the
// cluster has CTAs (16 x 33 KB, as a band is no lower than its halo; the count holds
// 2^20 - 1).
// (With a cluster barrier instead, whose release waits for the stores to be
// acknowledged, an exchange took about 0.8 us of a 400^2 lattice on 16 CTAs.)
template <int NT>
__device__ __forceinline__ void exchange_halos(uint32_t *lat, uint32_t lat_addr, int RW, int H, int D, int hmax, int block,
                                               Exchange &X)
{
    const int rw = D * RW;
    const uint32_t p = (uint32_t)block & 1u, phase = ((uint32_t)block >> 1) & 1u;
    uint32_t *const mbox = lat + (hmax + 2 * D) * RW + 2 * p * rw;
    const uint32_t mbox_addr = lat_addr + 4u * (uint32_t)((hmax + 2 * D) * RW + 2 * p * rw);
    if (X.arms != 0u) {
        if (X.arms & 1u) mbar_expect(exchange_bar(X.bar, 0u, p), 4u * (uint32_t)rw);
        if (X.arms & 2u) mbar_expect(exchange_bar(X.bar, 1u, p), 4u * (uint32_t)rw);
    }
    for (int idx = threadIdx.x; idx < 2 * rw; idx += NT) {
        const bool low = idx >= rw;  // the lowest rows go up (side 1 there), the highest down (side 0)
        const uint32_t v = lat[low ? D * RW + idx - rw : H * RW + idx];
        const uint32_t to = low ? X.to_prev : X.to_next;
        if (X.polls == kExchangePolls)
            store_counted(mbox_addr + 4u * (uint32_t)idx + to, v, exchange_bar(X.bar, low ? 1u : 0u, p) + to);
    }
    for (int idx = threadIdx.x; idx < 2 * rw; idx += NT) {
        const bool low = idx >= rw;
        if (!mbar_wait_cluster(exchange_bar(X.bar, low ? 1u : 0u, p), phase, X.polls)) {
            X.polls = 0;
            X.arms = 0u;
            break;
        }
        lat[low ? (D + H) * RW + idx - rw : idx] = mbox[idx];
    }
}

// Readies the mbarriers (before the cluster barrier that precedes the first exchange).
__device__ __forceinline__ void exchange_init(unsigned long long *xbar)
{
    if (threadIdx.x < kExchangeBars) mbar_init(smem_addr(xbar + threadIdx.x));
}

// halo_words: D * RW.  Side 0 is armed by the thread of the first word of a halo, side 1
// by that of the first word from below: the first that each waits for.
template <int NT>
__device__ __forceinline__ Exchange exchange_for(const unsigned long long *xbar, uint32_t lat_addr, int C, int rank,
                                                 int halo_words, bool withhold)
{
    return {smem_addr(xbar), mapa_distance(lat_addr, rank == 0 ? C - 1 : rank - 1),
            mapa_distance(lat_addr, rank + 1 == C ? 0 : rank + 1), withhold ? kExchangePollsShort : kExchangePolls,
            (threadIdx.x == 0 ? 1u : 0u) | ((int)threadIdx.x == halo_words % NT ? 2u : 0u)};
}

// By every thread after the last exchange.  A wait that ran out leaves a lattice that is no
// state of the chain: report it, and give stores in flight a second bounded wait.  No CTA
// leaves while a peer may still write into it.
__device__ __forceinline__ void exchange_end(const Exchange &X, bool withhold, long long *state)
{
    if (__syncthreads_or(X.polls == 0)) {
        if (threadIdx.x == 0) atomicExch((unsigned long long *)&state[kFault], 1ull);
        const int polls = withhold ? kExchangePollsShort : kExchangePolls;
        for (uint32_t i = 0; i < kExchangeBars; ++i)
            for (uint32_t par = 0; par < 2; ++par) mbar_wait_cluster(X.bar + 8u * i, par, polls);
    }
    cluster_barrier();
}
