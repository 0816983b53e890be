// Sixteen threads take and give back four words; no word has two holders.  Exit status 1 if one has.
#include <cstdio>
#include <vector>

#include "status_words.cuh"

int main() {
    soap::StatusWords<4> words;
    std::atomic<int> holders[4] = {};
    std::atomic<int> shared{0}, used{0};
    std::vector<std::thread> threads;
    for (int t = 0; t < 16; t++)
        threads.emplace_back([&] {
            for (int n = 0; n < 20000; n++) {
                const int i = words.claim();
                if (i < 0 || i >= 4 || holders[i].fetch_add(1) != 0) shared = 1;
                used |= 1 << i;
                if (n % 64 == 0) std::this_thread::yield();
                holders[i].fetch_sub(1);
                words.give_back(i);
            }
        });
    for (std::thread& t : threads) t.join();
    printf("%d %d\n", shared.load(), used.load());
    return shared.load();
}
