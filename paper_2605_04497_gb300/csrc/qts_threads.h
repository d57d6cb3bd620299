// Host threads of the table construction.
#pragma once

#include <exception>
#include <new>
#include <system_error>
#include <thread>
#include <vector>

namespace qts {

// fn(0) .. fn(n - 1), each on a thread of its own (shares before `own` on the caller's);
// shares whose thread cannot be started run on the caller's too.  An exception in
// any of them is thrown again here after all have ended: on its own thread it would
// end the process.
template <typename Fn>
void run_threads(int n, Fn&& fn, int own = 1) {
    std::vector<std::exception_ptr> thrown((size_t)n);
    auto call = [&](int k) noexcept {
        try {
            fn(k);
        } catch (...) {
            thrown[(size_t)k] = std::current_exception();
        }
    };
    std::vector<std::thread> th;
    th.reserve((size_t)n);
    int started = own;
    try {
        for (; started < n; ++started) th.emplace_back(call, started);
    } catch (const std::system_error&) {
    } catch (const std::bad_alloc&) {
    }
    for (int k = 0; k < own; ++k) call(k);
    for (int k = started; k < n; ++k) call(k);
    for (auto& x : th) x.join();
    for (auto& x : thrown)
        if (x) std::rethrow_exception(x);
}

}  // namespace qts
