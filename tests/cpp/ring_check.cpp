// Host check that a staging ring serves one scope at a time: a second thread's
// scope gets none while the first has it, the same thread's nested scope keeps
// it (under another ring it makes pageable copies), and it is free again after.
// No device is touched: the ring is never staged to.
#include <cstdio>
#include <new>
#include <thread>

#include "../../paper_1408_5092_gb300/csrc/core.h"

using namespace mpspt;

int main() {
    alignas(PinnedRing) unsigned char m1[sizeof(PinnedRing)] = {}, m2[sizeof(PinnedRing)] = {};
    auto* a = reinterpret_cast<PinnedRing*>(m1);   // members only, the constructor needs a device
    auto* b = reinterpret_cast<PinnedRing*>(m2);
    new (&a->taken) std::atomic<bool>(false);
    new (&b->taken) std::atomic<bool>(false);
    auto other = [](PinnedRing* r) {
        PinnedRing* got = r;
        std::thread([&] { RingScope s(r); got = thread_ring(); }).join();
        return got;
    };
    {
        RingScope s(a);
        if (thread_ring() != a || other(a) != nullptr || other(b) != b) { printf("second scope\n"); return 1; }
        {
            RingScope t(a);
            if (thread_ring() != a) { printf("nested\n"); return 1; }
            RingScope u(b);
            if (thread_ring() != b) return 1;
            RingScope v(a);
            if (thread_ring() != nullptr) { printf("nested under another\n"); return 1; }
        }
        if (thread_ring() != a || other(a) != nullptr || other(b) != b) { printf("after nesting\n"); return 1; }
    }
    if (thread_ring() != nullptr || other(a) != a) { printf("not released\n"); return 1; }
    printf("ok 1\n");
    return 0;
}
