// Host check of index and counting rules of the CUDA kernels (csrc/hostdev.h)
// that results on a GPU show only indirectly. Compiled with g++ by
// tests/test_hostdev_layout.py; prints "name value" lines.
#include <cstdio>

#include "hostdev.h"

using namespace hr;

// One to three rounds of arrivals at one counter, mixed (the units are alike,
// so their order does not matter), then a round by itself: it must have one
// last unit, the last to come, and leave the counter at zero.
static int arrival_violations() {
    int bad = 0;
    for (int units = 2; units <= 6; ++units) {
        unsigned counter = 0;
        auto inc = [&](unsigned most) {
            const unsigned old = counter;
            counter = old >= most ? 0 : old + 1;
            return old;
        };
        for (int mixed = units; mixed <= 3 * units; mixed += units) {      // one to three rounds before
            counter = 0;
            int lasts = 0;
            for (int i = 0; i < mixed; ++i) lasts += last_arrival(units, inc);
            if (lasts != mixed / units) ++bad;
            for (int i = 0; i < units; ++i)
                if (last_arrival(units, inc) != (i == units - 1)) ++bad;
            if (counter != 0) ++bad;
        }
    }
    return bad;
}

int main() {
    std::printf("arrival_violations %d\n", arrival_violations());
    return 0;
}
