// Host set-up over ranges of elements on several threads.
#pragma once

#include <algorithm>
#include <exception>
#include <new>
#include <system_error>
#include <thread>
#include <vector>

namespace esdg {

// work(e0, e1) over ranges of the K elements, on up to `most` threads of at least
// `least` elements.  A range whose thread cannot be started, or fails, is done by
// the calling thread, which passes on what that range throws then; every thread that
// was started is joined first.  (Thread: for the tests, a thread that cannot start.)
template <typename Thread = std::thread, typename F>
void in_threads(int K, int least, int most, F work) {
    int nt = std::max(1, std::min(most, (K + least - 1) / least));
    if (nt > 1) nt = std::max(1, std::min(nt, int(Thread::hardware_concurrency())));  // (10 us to ask)
    std::vector<char> done(nt, 0);
    auto range = [&](int t) {
        work(int((long long)K * t / nt), int((long long)K * (t + 1) / nt));
        done[t] = 1;
    };
    std::vector<Thread> pool;
    pool.reserve(nt);
    for (int t = 1; t < nt; ++t) {
        try {
            pool.emplace_back([&range, t] {
                try {
                    range(t);
                } catch (...) {  // (left to the calling thread)
                }
            });
        } catch (const std::system_error&) {  // no thread
            break;
        } catch (const std::bad_alloc&) {  // no memory for its state
            break;
        }
    }
    std::exception_ptr failed;
    try {
        range(0);
    } catch (...) {
        failed = std::current_exception();
    }
    for (auto& th : pool) th.join();
    if (failed) std::rethrow_exception(failed);
    for (int t = 1; t < nt; ++t)
        if (!done[t]) range(t);
}

}  // namespace esdg
