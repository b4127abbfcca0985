// Host program of test_sum.py: reads lines "n v1 .. vn" (hexadecimal doubles), writes the sum of each.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "dugks_sum.cuh"

int main() {
    int n;
    while (std::scanf("%d", &n) == 1) {
        std::vector<double> v(n);
        int top = 0;
        for (double &x : v) {
            if (std::scanf("%la", &x) != 1) return 1;
            top = std::max(top, dugks::exponent_of(x));
        }
        __int128 s = 0;
        for (double x : v) s += dugks::aligned(x, top);
        std::printf("%d %a\n", top >= dugks::SUM_LO && top < dugks::SUM_HI, dugks::unaligned(s, top));
    }
    return 0;
}
