// Host helpers of the C ABI (plain C++).
#pragma once
#include <cstdint>
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

// The cell of each of n particles from the starts [ncell + 1] of an image that
// may be damaged: false, and nothing written, unless they rise from 0 to n (a
// start beyond n followed by smaller ones would have keys written past the
// end).
inline bool keys_of_starts(const int *starts, int ncell, int64_t n, int *key)
{
    if (starts[0] != 0 || starts[ncell] != n) return false;
    for (int g = 0; g < ncell; ++g)
        if (starts[g + 1] < starts[g]) return false;
    for (int g = 0; g < ncell; ++g)
        for (int k = starts[g]; k < starts[g + 1]; ++k) key[k] = g;
    return true;
}

}  // namespace pic
