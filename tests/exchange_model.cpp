// The halo exchange of the resident sweeps (csrc/cluster_exchange.cuh), run on the host:
// every thread of every CTA of a cluster is a fiber, a store into another CTA is a message
// that lands when the scheduler lets it, and the mbarriers count arrivals and bytes as the
// PTX ISA defines them.  Adversaries hold back a warp or single stores for as long as
// anything else can move.  After every exchange each CTA's halo rows must be its
// neighbours' rows of that block, no wait may run out, and no arrival may meet a phase that
// has had its one.  When a store is lost, waits run out: the cluster must come to its end
// all the same, report it, and stay within the rules of the mbarriers.
#include <ucontext.h>

#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <functional>
#include <map>
#include <memory>
#include <random>
#include <vector>

#define KLMC_EXCHANGE_MODEL
#define __device__
#define __forceinline__ inline

namespace {

enum { kFault = 12 };
constexpr uint32_t kSpace = 1u << 20;  // a CTA's shared addresses start at a multiple of it

struct Bar {
    int pending = 0;
    long tx = 0;
    uint32_t phase = 0;
};

struct Message {
    uint32_t to, v, bar;
    int src;
    long number;
};

struct Cta {
    std::vector<uint32_t> smem;
    long long state[16] = {};
    int waiting = 0, generation = 0, vote = 0;
};

struct Fiber {
    ucontext_t uc;
    std::vector<char> stack;
    int cta = 0, tid = 0;
    bool done = false, gave_up = false, polling = false;
    std::function<bool()> ready;  // empty: may run
};

std::vector<Cta> ctas;
std::map<uint32_t, Bar> bars;
std::vector<Message> flying;
std::vector<std::unique_ptr<Fiber>> fibers;
Fiber *self = nullptr;
ucontext_t scheduler;
int threads = 0, cluster_waiting = 0, cluster_generation = 0;
long sent = 0, timeouts = 0, faults_found = 0;
bool rows_matter = true, withhold = false;
struct { unsigned x; } threadIdx;

void found(const char *what)
{
    if (faults_found++ == 0) std::printf("  %s\n", what);
}

// Gives way until ready() holds (at once: until the scheduler comes back); false when the
// scheduler found nothing else to do.
bool pause_until(std::function<bool()> ready)
{
    self->ready = std::move(ready);
    self->gave_up = false;
    swapcontext(&self->uc, &scheduler);
    self->ready = nullptr;
    return !self->gave_up;
}

void settle(Bar &b)
{
    if (b.tx <= -(1l << 20) || b.tx >= (1l << 20)) found("a byte count outside its range");
    if (b.pending == 0 && b.tx == 0) {
        b.pending = 1;
        b.phase += 1;
    }
}

uint32_t smem_addr(const void *p)
{
    for (size_t c = 0; c < ctas.size(); ++c) {
        const char *base = (const char *)ctas[c].smem.data();
        if ((const char *)p >= base && (const char *)p < base + 4 * ctas[c].smem.size())
            return (uint32_t)c * kSpace + (uint32_t)((const char *)p - base);
    }
    std::abort();
}

uint32_t mapa_distance(uint32_t addr, int rank) { return (uint32_t)rank * kSpace + addr % kSpace - addr; }

void mbar_init(uint32_t bar) { bars[bar] = Bar{1, 0, 0}; }

void mbar_expect(uint32_t bar, uint32_t bytes)
{
    pause_until(nullptr);
    Bar &b = bars.at(bar);
    if (b.pending != 1) found("an arrival on a phase that has had its one");
    b.tx += bytes;
    b.pending -= 1;
    settle(b);
}

void store_counted(uint32_t to, uint32_t v, uint32_t bar)
{
    pause_until(nullptr);
    if (to / kSpace != bar / kSpace || to / kSpace >= ctas.size() || to % kSpace + 4 > 4 * ctas[to / kSpace].smem.size())
        std::abort();
    flying.push_back({to, v, bar, self->cta, sent++});
}

bool mbar_wait_cluster(uint32_t bar, uint32_t parity, int)
{
    self->polling = true;
    const bool ok = pause_until([=] { return (bars.at(bar).phase & 1u) != parity; });
    self->polling = false;
    if (!ok) timeouts += 1;
    return ok;
}

void cta_barrier()
{
    Cta &c = ctas[self->cta];
    const int g = c.generation;
    if (++c.waiting == threads) {
        c.waiting = 0;
        c.generation += 1;
    }
    pause_until([g, &c] { return c.generation != g; });
}

void cluster_barrier()
{
    const int g = cluster_generation;
    if (++cluster_waiting == (int)fibers.size()) {
        cluster_waiting = 0;
        cluster_generation += 1;
    }
    pause_until([g] { return cluster_generation != g; });
}

int __syncthreads_or(int v)
{
    Cta &c = ctas[self->cta];
    c.vote |= v;
    cta_barrier();
    return c.vote;  // (one call in a run)
}

unsigned long long atomicExch(unsigned long long *p, unsigned long long v)
{
    const unsigned long long old = *p;
    *p = v;
    return old;
}

#include "cluster_exchange.cuh"

struct Shape {
    int C, H, D, RW, blocks;
};

uint32_t site(int cta, int row, int w, int block) { return (uint32_t)((((block * 16 + cta) * 64 + row) * 64 + w) * 2654435761u); }

// What a resident sweep does around the exchanges: phases of the band (here: new values
// for its rows), a barrier, the exchange, a barrier.
template <int NT>
void thread_main(const Shape &s)
{
    const int c = self->cta;
    Cta &cta = ctas[c];
    unsigned long long *const xbar = (unsigned long long *)cta.smem.data();
    uint32_t *const lat = cta.smem.data() + 16;
    exchange_init(xbar);
    cluster_barrier();
    Exchange X = exchange_for<NT>(xbar, smem_addr(lat), s.C, c, s.D * s.RW, withhold);
    const int prev = (c + s.C - 1) % s.C, next = (c + 1) % s.C;
    for (int b = 0; b < s.blocks; ++b) {
        for (int i = self->tid; i < s.H * s.RW; i += NT) lat[s.D * s.RW + i] = site(c, i / s.RW, i % s.RW, b);
        cta_barrier();
        exchange_halos<NT>(lat, smem_addr(lat), s.RW, s.H, s.D, s.H, b, X);
        cta_barrier();
        for (int i = self->tid; i < s.D * s.RW; i += NT) {
            const int r = i / s.RW, w = i % s.RW;
            if (!rows_matter) continue;
            if (lat[i] != site(prev, s.H - s.D + r, w, b)) found("a halo row that is not the upper neighbour's");
            if (lat[(s.D + s.H + r) * s.RW + w] != site(next, r, w, b)) found("a halo row that is not the lower neighbour's");
        }
        cta_barrier();
    }
    exchange_end(X, withhold, cta.state);
}

template <int NT>
void fiber_main(unsigned lo, unsigned hi)
{
    thread_main<NT>(*(const Shape *)((uintptr_t)lo | ((uintptr_t)hi << 32)));
    self->done = true;
    swapcontext(&self->uc, &scheduler);
}

enum Order { kAny, kOldestStore, kNewestStore };

// What becomes of the held stores when nothing else can move: they land, never do, or do
// after a wait or more has run out.
enum Held { kLate, kLost, kTooLate };

// Runs the cluster under one adversary; true when all went well.
template <int NT>
bool run(const Shape &s, std::function<bool(const Fiber &)> held_fiber, std::function<bool(const Message &)> held_store,
         Order order, unsigned seed, Held fate = kLate)
{
    rows_matter = fate == kLate;
    ctas.assign(s.C, Cta());
    bars.clear();
    flying.clear();
    fibers.clear();
    threads = NT;
    cluster_waiting = cluster_generation = 0;
    sent = timeouts = faults_found = 0;
    for (Cta &c : ctas) c.smem.assign(16 + (size_t)s.RW * (s.H + 6 * s.D), 0u);
    for (int c = 0; c < s.C; ++c)
        for (int t = 0; t < NT; ++t) {
            fibers.emplace_back(new Fiber);
            Fiber &f = *fibers.back();
            f.cta = c;
            f.tid = t;
            f.stack.resize(32 << 10);
            getcontext(&f.uc);
            f.uc.uc_stack.ss_sp = f.stack.data();
            f.uc.uc_stack.ss_size = f.stack.size();
            f.uc.uc_link = nullptr;
            const uintptr_t p = (uintptr_t)&s;
            makecontext(&f.uc, (void (*)())fiber_main<NT>, 2, (unsigned)p, (unsigned)((unsigned long long)p >> 32));
        }
    std::mt19937 rng(seed);
    auto step = [&](Fiber *f) {
        self = f;
        threadIdx.x = (unsigned)f->tid;
        swapcontext(&scheduler, &f->uc);
    };
    auto land = [&](size_t i) {
        const Message m = flying[i];
        flying.erase(flying.begin() + (long)i);
        ctas[m.to / kSpace].smem[m.to % kSpace / 4] = m.v;
        Bar &b = bars.at(m.bar);
        b.tx -= 4;
        settle(b);
    };
    while (true) {
        std::vector<Fiber *> free, held;
        bool all_done = true;
        for (auto &f : fibers) {
            if (f->done) continue;
            all_done = false;
            if (f->ready && !f->ready()) continue;
            (held_fiber && held_fiber(*f) ? held : free).push_back(f.get());
        }
        if (all_done) break;
        std::vector<size_t> stores, held_stores;
        for (size_t i = 0; i < flying.size(); ++i) (held_store && held_store(flying[i]) ? held_stores : stores).push_back(i);
        if (!stores.empty() && (free.empty() || rng() % 2)) {
            land(order == kOldestStore ? stores.front() : (order == kNewestStore ? stores.back() : stores[rng() % stores.size()]));
        } else if (!free.empty()) {
            step(free[rng() % free.size()]);
        } else if (!held.empty()) {
            step(held[rng() % held.size()]);
        } else if (!held_stores.empty() && (fate == kLate || (fate == kTooLate && timeouts > 0 && rng() % 4 == 0))) {
            land(held_stores[rng() % held_stores.size()]);
        } else {  // nothing can move: a wait runs out
            std::vector<Fiber *> polling;
            for (auto &f : fibers)
                if (!f->done && f->polling) polling.push_back(f.get());
            if (polling.empty()) {
                found("threads that wait at a barrier for ever");
                return false;
            }
            Fiber *const f = polling[rng() % polling.size()];
            f->gave_up = true;
            step(f);
        }
    }
    int reports = 0;
    for (Cta &c : ctas) reports += c.state[kFault] != 0;
    if (fate == kLate && (timeouts > 0 || reports > 0)) found("a wait that nothing ends");
    if (withhold && (sent > 0 || reports < s.C)) found("stores sent, or a CTA without a report, under the test hook");
    if (fate != kLate && (timeouts == 0 || reports == 0)) found("a wait that ran out and nobody reports");
    return faults_found == 0;
}

int failures = 0;

void check(bool ok, const char *what, const Shape &s, int NT, int a, int b)
{
    if (ok) return;
    std::printf("FAILED: %s (%d, %d) with %d CTAs of %d threads, %d rows, halo %d x %d\n", what, a, b, s.C, NT, s.H, s.D, s.RW);
    failures += 1;
}

template <int NT>
void all_adversaries(const Shape &s)
{
    for (unsigned seed = 0; seed < 4; ++seed) {
        check(run<NT>(s, nullptr, nullptr, kAny, seed), "stores land at random, seed", s, NT, (int)seed, 0);
        check(run<NT>(s, nullptr, nullptr, kNewestStore, seed), "newest store first, seed", s, NT, (int)seed, 0);
    }
    for (int c = 0; c < s.C; ++c)
        for (int w = 0; w < NT / 32; ++w)
            check(run<NT>(s, [=](const Fiber &f) { return f.cta == c && f.tid / 32 == w; }, nullptr, kOldestStore, 7),
                  "a warp held back: CTA, warp", s, NT, c, w);
    withhold = true;
    check(run<NT>(s, nullptr, nullptr, kAny, 0, kLost), "stores withheld", s, NT, 0, 0);
    withhold = false;
    const long all = (long)s.C * s.blocks * 2 * s.D * s.RW;
    std::mt19937 rng(11);
    for (int k = 0; k < 12; ++k) {
        const long n = (long)(rng() % (unsigned long)all);
        check(run<NT>(s, nullptr, [=](const Message &m) { return m.number == n; }, kOldestStore, (unsigned)k),
              "a store held back: number", s, NT, (int)n, 0);
        const long few = n % (2l * s.C * 2 * s.D * s.RW);  // of the first two blocks
        check(run<NT>(s, nullptr, [=](const Message &m) { return m.number == few; }, kOldestStore, (unsigned)k, kLost),
              "a store lost: number", s, NT, (int)few, 0);
        check(run<NT>(s, nullptr, [=](const Message &m) { return m.number >= few && m.number < few + 40; }, kAny, (unsigned)k,
                      kTooLate),
              "stores too late: from number", s, NT, (int)few, 0);
    }
}

}  // namespace

int main()
{
    all_adversaries<64>({3, 6, 4, 8, 5});   // either side's rows are one warp's
    all_adversaries<64>({2, 10, 4, 8, 5});  // both neighbours are the same CTA
    all_adversaries<96>({4, 5, 5, 9, 4});   // more than one pass of the threads, a remainder
    std::printf(failures ? "%d adversaries won\n" : "the exchange holds\n", failures);
    return failures != 0;
}
