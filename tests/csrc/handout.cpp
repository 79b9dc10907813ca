// Test harness (host only): runs take_work (pv_handout.cuh) with the warps of a CTA emulated lane by lane, one
// thread each, so the CPU tests can check the hand-out of chains without a GPU. Warp-wide operations meet at a
// barrier of the warp's lanes; between them the lanes run freely, as the hardware allows.
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <mutex>
#include <thread>
#include <vector>

#include <cuda_runtime.h>

#define PV_FULL 0xffffffffu

namespace emu {
struct Parted {};            // lanes of a warp that wait at different places
struct Warp {
    std::mutex m;
    std::condition_variable cv;
    int waiting = 0;
    unsigned long long turn = 0;
    unsigned long long value[32];
    void meet() {
        std::unique_lock<std::mutex> l(m);
        const unsigned long long mine = turn;
        if (++waiting == 32) {
            waiting = 0;
            ++turn;
            cv.notify_all();
        } else {
            if (!cv.wait_for(l, std::chrono::seconds(10), [&] { return turn != mine; })) throw Parted();
        }
    }
};
struct Index { int x; };
static thread_local Index threadIdx;
static thread_local Warp* warp;
static std::atomic<unsigned long long> clock_ns{1};
static int lane() { return threadIdx.x & 31; }
// Lanes go on from a shuffle at times of their own.
static void stray() {
    static thread_local unsigned n = 12345u + 977u * threadIdx.x;
    n = n * 1664525u + 1013904223u;
    if ((n >> 29) == 0) std::this_thread::sleep_for(std::chrono::microseconds(60));
}
}  // namespace emu

using emu::threadIdx;

template <class T>
static T __shfl_sync(unsigned, T v, int src) {
    emu::warp->value[emu::lane()] = (unsigned long long)v;
    emu::warp->meet();
    const T r = (T)emu::warp->value[src];
    emu::warp->meet();
    emu::stray();
    return r;
}
static unsigned __ballot_sync(unsigned, bool v) {
    emu::warp->value[emu::lane()] = v;
    emu::warp->meet();
    unsigned r = 0;
    for (int i = 0; i < 32; ++i) r |= (unsigned)emu::warp->value[i] << i;
    emu::warp->meet();
    return r;
}
static void __syncwarp() { emu::warp->meet(); }
static void __threadfence_block() { std::atomic_thread_fence(std::memory_order_seq_cst); }
static void __nanosleep(unsigned) { std::this_thread::yield(); }
static int __ffs(unsigned v) { return __builtin_ffs((int)v); }
static int min(int a, int b) { return a < b ? a : b; }
static int atomicCAS(int* p, int expect, int v) {
    __atomic_compare_exchange_n(p, &expect, v, false, __ATOMIC_SEQ_CST, __ATOMIC_SEQ_CST);
    return expect;
}
static int atomicExch(int* p, int v) { return __atomic_exchange_n(p, v, __ATOMIC_SEQ_CST); }
static int atomicAdd(int* p, int v) { return __atomic_fetch_add(p, v, __ATOMIC_SEQ_CST); }
static int atomicSub(int* p, int v) { return __atomic_fetch_sub(p, v, __ATOMIC_SEQ_CST); }
static int atomicOr(int* p, int v) { return __atomic_fetch_or(p, v, __ATOMIC_SEQ_CST); }
static unsigned long long globaltimer() { return emu::clock_ns.load(); }

#include "pv_handout.cuh"

namespace {

void clear(pv::CtaWork& w) {
    w.lock = w.done = w.next = w.count = 0;
    w.pending = -1;
    w.blk = w.pos = w.pair = w.unit0 = w.slot = 0;
    for (int k = 0; k < pv::kLigSlots; ++k) {
        w.lig[k] = -1;
        w.refs[k] = w.ready[k] = 0;
    }
}

struct Job {
    std::vector<int> order;
    std::vector<PvPairDesc> pairs;
    int queue = 0, err = 0;
    pv::SearchArgs A{};
    pv::CtaWork W{};
    // a pair per ligand, blocks x units of each
    Job(int n_ligs, int blocks, int units, int item_units, int slots, unsigned long long wait_ns) {
        for (int i = 0; i < n_ligs; ++i) {
            order.push_back(i);
            pairs.push_back(PvPairDesc{i, 0, 0, i});
        }
        A.order = order.data();
        A.pairs = pairs.data();
        A.queue = &queue;
        A.err = &err;
        A.units = units;
        A.item_units = item_units;
        A.items_per_pair = (units + item_units - 1) / item_units;
        A.items_per_block = A.items_per_pair * n_ligs;
        A.n_items = blocks * A.items_per_block;
        A.lig_slots = slots;
        A.wait_ns = wait_ns;
        clear(W);
    }
};

// Runs the warps; returns whether lanes of one parted.
template <class F>
bool run_warps(int n, F&& body) {
    std::atomic<bool> parted{false};
    std::vector<emu::Warp> warps(n);
    std::vector<std::thread> lanes;
    for (int t = 0; t < 32 * n; ++t)
        lanes.emplace_back([&, t] {
            threadIdx.x = t;
            emu::warp = &warps[t / 32];
            try {
                body(t / 32, t % 32);
            } catch (const emu::Parted&) {
                parted = true;
            }
        });
    for (std::thread& t : lanes) t.join();
    return parted;
}

bool same(const pv::WarpWork& a, const pv::WarpWork& b) {
    return a.status == b.status && a.blk == b.blk && a.pos == b.pos && a.pair == b.pair && a.unit == b.unit && a.slot == b.slot;
}

}  // namespace

// Warps of one CTA work a whole job off. out = units handed out once, units in all, takes whose lanes disagreed,
// units whose slot held another ligand while they ran, error bits.
extern "C" void handout_job(int warps, int n_ligs, int blocks, int units, int item_units, int slots, int* out) {
    Job J(n_ligs, blocks, units, item_units, slots, 30000000000ull);
    std::vector<std::atomic<int>> taken(blocks * n_ligs * units);
    std::atomic<int> staged[pv::kLigSlots], split{0}, wrong{0};
    for (auto& s : staged) s = -1;
    std::vector<std::vector<pv::WarpWork>> seen(warps, std::vector<pv::WarpWork>(32));
    std::atomic<bool> stop{false};
    const bool parted = run_warps(warps, [&](int warp, int lane) {
        for (unsigned n = 1;; ++n) {
            const pv::WarpWork w = pv::take_work(J.A, J.W);
            seen[warp][lane] = w;
            emu::warp->meet();
            bool agree = true;
            for (int i = 1; i < 32; ++i) agree = agree && same(seen[warp][0], seen[warp][i]);
            emu::warp->meet();
            if (!agree) {                     // the lanes would run on different records: end the job
                if (lane == 0) ++split;
                stop = true;
            }
            if (!agree || w.status == 0 || stop) {
                emu::warp->meet();
                return;
            }
            if (lane == 0) {
                ++taken[(w.blk * n_ligs + w.pos) * units + w.unit];
                const int lig = J.pairs[w.pair].ligand;
                if (w.status == 2) {
                    staged[w.slot] = lig;
                    atomicExch(&J.W.ready[w.slot], 1);
                } else {
                    while (!stop && !__atomic_load_n(&J.W.ready[w.slot], __ATOMIC_SEQ_CST)) std::this_thread::yield();
                }
                const int spins = (int)((n * 2654435761u + warp * 40503u) >> 20) & 255;
                for (int i = 0; i < spins; ++i) {
                    if (staged[w.slot] != lig) ++wrong;
                    std::this_thread::yield();
                }
                atomicSub(&J.W.refs[w.slot], 1);
            }
            emu::warp->meet();
        }
    });
    int once = 0;
    for (auto& t : taken) once += t == 1;
    out[0] = once;
    out[1] = (int)taken.size();
    out[2] = split + parted;
    out[3] = wrong;
    out[4] = J.err;
}

// Warp 0 works for busy_ns (by the emulated clock) on the one ligand slot while warp 1 waits for it with another
// ligand, of two units of two ligands. out = units that warp 1 took, units taken, error bits.
extern "C" void handout_starved(unsigned long long busy_ns, unsigned long long wait_ns, int* out) {
    Job J(2, 1, 1, 1, 1, wait_ns);
    emu::clock_ns = 1000;
    std::atomic<int> taken[2] = {{0}, {0}};
    std::atomic<bool> held{false}, gone{false};
    run_warps(2, [&](int warp, int lane) {
        if (warp == 1 && lane == 0)
            while (!held) std::this_thread::yield();
        emu::warp->meet();
        for (;;) {
            const pv::WarpWork w = pv::take_work(J.A, J.W);
            if (w.status == 0) {
                if (warp == 1) gone = true;
                return;
            }
            if (lane == 0) {
                ++taken[warp];
                if (warp == 0 && !held) {
                    held = true;
                    while (__atomic_load_n(&J.W.pending, __ATOMIC_SEQ_CST) < 0) std::this_thread::yield();
                    for (int i = 0; i < 50; ++i) {         // the clock runs on while warp 1 looks at it
                        emu::clock_ns += busy_ns / 50;
                        std::this_thread::sleep_for(std::chrono::milliseconds(10));
                    }
                }
                atomicSub(&J.W.refs[w.slot], 1);
                while (warp == 0 && !taken[1] && !gone) std::this_thread::yield();   // warp 1 chooses first
            }
            emu::warp->meet();
        }
    });
    out[0] = taken[1];
    out[1] = taken[0] + taken[1];
    out[2] = J.err;
}

extern "C" int handout_step_block(int steps, int fixed_cta, int all_resident, int items_per_block) {
    return pv::step_block(steps, fixed_cta, all_resident, items_per_block);
}
