// decode_node() (dp_device.cuh) on the CPU, for every number of mass nodes and
// nodes at both ends of lines all over the range of a node index.  Prints the
// nodes decoded and the ones decoded wrongly.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "cuda_on_host.h"

#include "dp_device.cuh"

using namespace dpk;

int main()
{
    long long looked = 0, wrong = 0;
    std::vector<unsigned> lines(1);
    for (int n_m = 2; n_m <= 1024; ++n_m) {
        Geo<double> g;
        memset(&g, 0, sizeof g);
        g.n_m = n_m;
        line_divisor(n_m, g.line_mul, g.line_shift);
        const long long last = 2147483646LL / n_m;
        for (int k = 0; k < 4000; ++k) {
            // lines: the first, the last, around each power of two, evenly in between
            long long line = k < 1000 ? last * k / 999 : k < 2000 ? (1LL << (k % 31)) + k % 7 - 3 : last - (k - 2000);
            line = std::min(std::max(line, 0LL), last);
            for (int m : {0, 1, n_m / 2, n_m - 1}) {
                const long long j = line * n_m + m;
                if (j > 2147483646LL) continue;
                // decode_node() looks its line up: a table of one entry at that line's place
                g.lines = lines.data() - line;
                lines[0] = (unsigned)(line % 1024) | (unsigned)(line % 1000) << 10 | (unsigned)(line % 999) << 20;
                const unsigned got = __umulhi((unsigned)j, g.line_mul) >> g.line_shift;
                ++looked;
                if (got != (unsigned)line) {   // not decoded: the table has this line only
                    ++wrong;
                    continue;
                }
                int i[4];
                decode_node(g, (int)j, i);
                wrong += i[3] != m || i[0] != line % 1024 || i[1] != line % 1000 || i[2] != line % 999;
            }
        }
    }
    printf("%lld %lld\n", looked, wrong);
    return 0;
}
