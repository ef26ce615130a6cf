// Host check of the block-wide bounded wait (bounded_wait.cuh) with threads in
// the part of a block's: a condition that never comes true ends every thread's
// wait with false; one that comes true before, around or after the limit ends
// all threads' waits alike, leaves the counter at 0 when they succeed, and the
// next wait starts afresh.  And of the inner solver's status words: a wait that
// gave up is a timeout, not a breakdown.
// Prints "ok <cases>" and exits 0, or reports the first violation and exits 1.
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>

#include "../paper_2104_04609_gb300/csrc/bounded_wait.cuh"
#include "../paper_2104_04609_gb300/csrc/osrc_internal.cuh"

static unsigned long long ns() {
    return (unsigned long long)std::chrono::duration_cast<std::chrono::nanoseconds>(
               std::chrono::steady_clock::now().time_since_epoch())
        .count();
}

struct Count {
    std::atomic<int> *c;
    int load() const { return c->load(); }
    void add() const { c->fetch_add(1); }
    bool cas(int e, int v) const { return c->compare_exchange_strong(e, v); }
};

struct Barrier {  // of n threads, reusable
    std::atomic<int> in{0}, gen{0};
    int n;
    explicit Barrier(int n_) : n(n_) {}
    void wait() {
        const int g = gen.load();
        if (in.fetch_add(1) + 1 == n) {
            in.store(0);
            gen.fetch_add(1);
        } else {
            while (gen.load() == g) std::this_thread::yield();
        }
    }
};

int main() {
    constexpr int N = 4, WAITS = 3;
    constexpr unsigned long long LIMIT = 200000;  // 0.2 ms
    int cases = 0, all_true = 0, all_false = 0;
    for (int rep = 0; rep < 400; ++rep) {
        // the condition of wait w comes true delay ns after its start (0: at once, < 0: never)
        const long long at = rep % 4 == 0 ? -1 : (long long)LIMIT * (rep % 100) / 50;
        std::atomic<int> count{0};
        std::vector<std::atomic<int>> ready(WAITS);
        for (auto &r : ready) r.store(0);
        std::vector<int> res(N * WAITS, -1);
        Barrier bar(N + 1);
        std::vector<std::thread> th;
        std::atomic<bool> stop{false};  // a failed wait is the block's last
        for (int t = 0; t < N; ++t)
            th.emplace_back([&, t] {
                for (int w = 0; w < WAITS; ++w) {
                    bar.wait();
                    if (stop.load()) return;
                    res[t * WAITS + w] = bounded_wait([&] { return ready[w].load() != 0; }, ns, Count{&count}, N, LIMIT);
                    bar.wait();
                }
            });
        bool fail = false;
        for (int w = 0; w < WAITS; ++w) {
            bar.wait();
            if (stop.load()) break;
            if (at >= 0) {
                const unsigned long long t0 = ns();
                while (ns() - t0 < (unsigned long long)at) std::this_thread::yield();
                ready[w].store(1);
            }
            bar.wait();
            int ok = 0;
            for (int t = 0; t < N; ++t) ok += res[t * WAITS + w];
            ++cases;
            (ok ? all_true : all_false)++;
            if (ok != 0 && ok != N) fail = true, std::printf("FAIL rep %d wait %d: %d of %d threads succeeded\n", rep, w, ok, N);
            if (at < 0 && ok) fail = true, std::printf("FAIL rep %d: a wait for nothing succeeded\n", rep);
            if (at == 0 && !ok) fail = true, std::printf("FAIL rep %d: a condition that was true failed\n", rep);
            if (!ok || fail) stop.store(true);
        }
        for (auto &t : th) t.join();
        if (fail) return 1;
        if (!stop.load() && count.load() != 0) {
            std::printf("FAIL rep %d: counter %d after successful waits\n", rep, count.load());
            return 1;
        }
    }
    if (all_true < 100 || all_false < 100) {
        std::printf("FAIL only %d successful and %d failed waits met\n", all_true, all_false);
        return 1;
    }
    int worst = 3;
    const int fine[] = {5, 0, 9, 2}, open_[] = {5, -7, 2}, broke[] = {1, -1000004, -3}, lost[] = {1, KRY_LOST, -3},
              big[] = {-2100000000};
    if (kry_stat_code(fine, 4, &worst) != OSRC_OK || worst != 9) return std::printf("FAIL status ok\n"), 1;
    if (kry_stat_code(open_, 3, &worst) != OSRC_NOT_CONVERGED) return std::printf("FAIL status -7\n"), 1;
    if (kry_stat_code(broke, 3, &worst) != OSRC_BREAKDOWN) return std::printf("FAIL status breakdown\n"), 1;
    if (kry_stat_code(lost, 3, &worst) != OSRC_TIMEOUT) return std::printf("FAIL status lost\n"), 1;
    if (kry_stat_code(big, 1, &worst) != OSRC_BREAKDOWN) return std::printf("FAIL status many iterations\n"), 1;
    std::printf("ok %d\n", cases);
    return 0;
}
