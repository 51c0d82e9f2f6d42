// Host-only check that building the separable path's tables for a new slope holds up nobody who
// asks for another one (paper_2103_09686_gb300/csrc/sep_basis.cpp).  Prints the time of the build and the
// longest wait of a second thread for a slope that is there; exits 1 when that is more than half
// the build, or when two threads asking for the same new slope get different tables.
#include <stdio.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <thread>

#include "sep_basis.h"

static double now() {
    return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

int main() {
    dmcr::sep_basis(10.f);
    bool ok = true;
    for (int i = 0; i < 3; ++i) {                       // the best of three: a busy machine
        std::atomic<bool> started{false}, done{false};
        std::shared_ptr<const dmcr::SepBasis> a, b;
        double build = 0.0;
        std::thread first([&] {
            const double t = now();
            started = true;
            a = dmcr::sep_basis(15.f + (float)i);
            build = now() - t;
            done = true;
        });
        std::thread same([&] { b = dmcr::sep_basis(15.f + (float)i); });
        while (!started) std::this_thread::yield();
        double longest = 0.0;
        while (!done) {
            const double t = now();
            dmcr::sep_basis(10.f);
            longest = std::max(longest, now() - t);
        }
        first.join();
        same.join();
        printf("build %.3f s, longest wait %.6f s\n", build, longest);
        if (a != b) return 1;
        ok = longest < 0.5 * build;
        if (ok) break;
    }
    return ok ? 0 : 1;
}
