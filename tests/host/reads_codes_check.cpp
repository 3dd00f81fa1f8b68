// Host-only check of reads_codes_early: of the batches the decode kernel may take,
// only those that the library has always run in a kernel that reads codes ahead of
// stream order (4 bits up to 7 rows, 3 and 8 bits up to 4) may do so; a larger batch
// may follow, in stream order, a kernel that writes its codes.  Prints "ok" or the
// first failing case.
#include <stdio.h>

#include "internal.h"

int main()
{
    const int widths[3] = {3, 4, 8};
    for (int bits : widths)
        for (int64_t B = 1; B <= 40; ++B) {
            const bool may = B <= 4 || (bits == 4 && B < 8);
            if (logq::reads_codes_early(bits, B) && !may) {
                printf("fail bits=%d B=%d\n", bits, (int)B);
                return 1;
            }
        }
    printf("ok\n");
    return 0;
}
