// Host check of the two-pass kernels' chunk plan (march_plan.h): "nx ny nz pad" lines in, the predictor's and the
// corrector's chunk out (152 SMs); with the argument "sweep", every plan of a range of grids must lie in [1, planes].
#include <cstdio>
#include <cstring>
#include <initializer_list>

#include "march_plan.h"

using namespace rhd;

int main(int argc, char** argv)
{
    if (argc > 1 && !std::strcmp(argv[1], "sweep")) {
        long long bad = 0, n = 0;
        for (int planes = 3; planes <= 600; planes = planes < 40 ? planes + 1 : planes + 7)
            for (long long tiles = 1; tiles <= 2000000; tiles = tiles < 64 ? tiles + 1 : tiles * 3 / 2)
                for (int sms : {1, 8, 152}) {
                    for (const MarchCost& m : {kMarchPred, kMarchCorr}) {
                        const int c = march_chunk(m, tiles, planes, sms);
                        bad += c < 1 || c > planes;
                        ++n;
                    }
                }
        std::printf("%lld %lld\n", bad, n);
        return 0;
    }
    int x, y, z, p;
    while (std::scanf("%d %d %d %d", &x, &y, &z, &p) == 4)
        std::printf("%d %d\n", march_chunk(kMarchPred, (long long)((x + 2 * p + 31) / 32) * ((y + 2 * p + 7) / 8), z + 2 * p, 152),
                    march_chunk(kMarchCorr, (long long)((x + 31) / 32) * ((y + 7) / 8), z, 152));
    return 0;
}
