// PerDevice: a value of one device is not another's, a search that failed is made again, and
// a value found is not searched for twice, by any number of threads.
// OnDevice: the device is current inside, and the one before is afterwards.
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>

#include "ptebd_device.h"

#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)

struct Fake {
    int* current;
    int* sets;
    int refuse;  // a device that cannot be made current
    int get(int* d) { *d = *current; return 0; }
    int set(int d) { ++*sets; if (d == refuse) return 101; *current = d; return 0; }
};

int on_device() {
    int current = 0, sets = 0;
    {
        ptebd::OnDevice<Fake> here(0, Fake{&current, &sets, -1});
        CHECK(here.error() == 0 && current == 0);
    }
    CHECK(sets == 0);  // (the usual case: nothing to do)
    {
        ptebd::OnDevice<Fake> there(1, Fake{&current, &sets, -1});
        CHECK(there.error() == 0 && current == 1);
    }
    CHECK(current == 0 && sets == 2);
    {
        ptebd::OnDevice<Fake> there(3, Fake{&current, &sets, 3});
        CHECK(there.error() == 101 && current == 0);
    }
    CHECK(current == 0 && sets == 3);
    return 0;
}

int main() {
    if (on_device()) return 1;
    ptebd::PerDevice<const void*, int> counts;
    int key_a = 0, key_b = 0, searches = 0;
    auto finds = [&](int v) { return [&searches, v](int* out) { ++searches; *out = v; return 0; }; };
    auto fails = [&](int* out) { ++searches; *out = 7; return 2; };

    CHECK(counts.get(0, &key_a, fails) == 0);         // (nothing of a failed search comes back)
    CHECK(counts.get(0, &key_a, finds(152)) == 152);  // and none is kept
    CHECK(counts.get(1, &key_a, finds(76)) == 76);    // another device
    CHECK(counts.get(0, &key_b, finds(9)) == 9);      // another kernel
    CHECK(searches == 4);
    CHECK(counts.get(0, &key_a, finds(-1)) == 152);
    CHECK(counts.get(1, &key_a, finds(-1)) == 76);
    CHECK(searches == 4);

    std::atomic<int> made{0}, wrong{0};
    std::vector<std::thread> threads;
    for (int t = 0; t < 16; ++t)
        threads.emplace_back([&, t] {
            for (int d = 0; d < 50; ++d)
                if (counts.get(2 + d, &key_a, [&](int* out) { ++made; *out = 1000 + d; return 0; }) != 1000 + d) ++wrong;
        });
    for (auto& t : threads) t.join();
    CHECK(made == 50 && wrong == 0);
    return 0;
}
