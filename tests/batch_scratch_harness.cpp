// Test harness for the scratch of a batch plan's split classes
// (host_sched.h): reads "capacity streams classes" and a line "stream per_pair
// count wave" per class, takes the scratch from an allocator of that capacity,
// and prints whether it fits, the bytes still allocated, every class's wave
// and every stream's bytes.
#include <iostream>
#include <map>
#include <vector>

#include "../paper_1005_1497_gb300/csrc/host_sched.h"

int main()
{
    size_t capacity = 0, classes = 0;
    int streams = 0;
    std::cin >> capacity >> streams >> classes;
    std::vector<ntt::ScratchClass> c(classes);
    for (auto &x : c) std::cin >> x.stream >> x.per_pair >> x.count >> x.least;
    std::map<size_t, size_t> held;                      // address -> bytes
    size_t used = 0, next = 256;
    auto alloc = [&](size_t bytes) -> void * {
        if (used + bytes > capacity) return nullptr;
        used += bytes;
        held[next] = bytes;
        return (void *)(next++);
    };
    auto release = [&](void *p) {
        used -= held.at((size_t)p);
        held.erase((size_t)p);
    };
    std::vector<void *> pieces(streams, nullptr);
    const bool ok = ntt::take_scratch(c, pieces, alloc, release);
    std::cout << ok << " " << used;
    for (auto &x : c) std::cout << " " << x.wave;
    for (void *p : pieces) std::cout << " " << (p ? held.at((size_t)p) : 0);
    std::cout << "\n";
    return 0;
}
