// Host-only check of reads_codes_early: of the batches the decode kernel may take, only
// those may read codes ahead of stream order that the library has always run in a kernel
// that does.  Those are 3 and 8 bits up to 4 rows, 4 bits up to 7, and 4 bits up to 16
// wherever the time model of the workspace sizes keeps off the tensor-core launch: here
// for every number of rows and k of a fine grid, with that launch's estimate bounded from
// below (one round of CTAs, whole or split k ranges of at least 8 steps).  A larger batch may
// follow, in stream order, a kernel that writes its codes.  Prints "ok" or the first
// failing case.
#include <stdio.h>

#include "internal.h"

int main()
{
    const int widths[3] = {3, 4, 8};
    for (int bits : widths)
        for (int64_t B = 1; B <= 40; ++B)
            for (int64_t K = 128; K <= 65536; K += K < 2048 ? 128 : K / 2048 * 128)
                for (int64_t N = 1; N <= 1 << 20; N += 1 + N / 16) {
                    bool may = B <= 4 || (bits == 4 && B < 8);
                    if (bits == 4 && B >= 8 && B <= 16) {
                        // steps of the longest CTA on 152 SMs, 0.5 us each, and 6 to fill and drain
                        const double tiles = (double)((N + 127) / 128), steps = (double)K / 64;
                        const double share = tiles * steps / 152 > 1 ? tiles * steps / 152 : 1;
                        const double whole = 0.5 * ((steps > share ? steps : share) + 6) + 3;
                        const double split = 0.5 * ((share > 8 ? share : 8) + 6 + 6) + 3;
                        const double cores = (double)N * (double)K * (B <= 8 ? 0.46e-6 : 0.84e-6) + 2;
                        may = cores <= (whole < split ? whole : split);
                    }
                    if (logq::reads_codes_early(bits, B, N * K) && !may) {
                        printf("fail bits=%d B=%d N=%ld K=%ld\n", bits, (int)B, (long)N, (long)K);
                        return 1;
                    }
                }
    printf("ok\n");
    return 0;
}
