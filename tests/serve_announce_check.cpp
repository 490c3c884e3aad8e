// The scheduler announces every request of a group before any of them runs, so that an
// executor that merges their work knows whom to wait for, however late a companion's
// thread starts.  One worker, held by another request while four mergeable REBUILDs queue up.
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>

#include "serve_core.h"

using namespace lace_serve;

struct Exec {
    struct Handle {};
    std::atomic<int> announced{0}, early{0}, ran{0};

    size_t predict(const SystemDesc&, const Handle&, int, int) { return 1; }
    size_t held(const Handle&) { return 1; }
    void release(Handle&) {}
    int merge_key(const SystemDesc& d) const { return d.flags; }
    void announce(const SystemDesc& d, Request& r) {
        r.announced = d.flags;
        if (d.flags) ++announced;
    }
    void withdraw(const SystemDesc&, Request& r) {
        if (r.announced) --announced;
        r.announced = 0;
    }
    int run(const SystemDesc& d, Handle&, Request& r) {
        if (!d.flags) {
            std::this_thread::sleep_for(std::chrono::milliseconds(50));
            return S_OK;
        }
        if (announced.load() != 4 || r.announced != d.flags) ++early;
        ++ran;
        return S_OK;
    }
};

int main() {
    Exec ex;
    {
        Scheduler<Exec> s(ex, 1, 1, 100);
        s.set_rebuild_group(4);
        std::vector<long long> ids;
        double in = 0.0, out = 0.0;
        for (int k = 0; k < 5; ++k) {
            const int sys = s.add_system(SystemDesc{{10, 10, 10}, {48, 48, 48}, 10.0, 1, 0, 0.0, k ? 48 : 0});
            long long id = -1;
            if (s.submit(sys, REQ_REBUILD, &in, 1, &out, &id) != S_OK) return 2;
            ids.push_back(id);
        }
        for (long long id : ids) {
            int done = 0, result = 0;
            double lat = 0.0, e = 0.0;
            long long np = 0;
            s.poll(id, true, &done, &result, &lat, &e, &np);
        }
    }
    std::printf("announced %d, ran %d, before all were announced %d\n", ex.announced.load(), ex.ran.load(), ex.early.load());
    return ex.announced.load() == 4 && ex.ran.load() == 4 && ex.early.load() == 0 ? 0 : 1;
}
