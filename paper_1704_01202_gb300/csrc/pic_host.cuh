// Host helpers of the C ABI (plain C++).
#pragma once
#include <thread>
#include <vector>

namespace pic {

// f(0) .. f(shares - 1), a host thread each, the calling thread among them.
// Where no more threads are to be had (a process or memory limit), the calling
// thread takes the shares that are left: the call does not depend on them, and
// no exception leaves it with threads still running (which would end the
// process).  f does not throw.
template <class F>
void host_shares(int shares, const F &f)
{
    std::vector<std::thread> th;
    int started = 1;
    try {
        th.reserve(shares);
        for (; started < shares; ++started) th.emplace_back([&f, started] { f(started); });
    } catch (...) {
    }
    if (shares > 0) f(0);
    for (int t = started; t < shares; ++t) f(t);
    for (auto &x : th) x.join();
}

}  // namespace pic
