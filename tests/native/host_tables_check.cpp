// Host-only check of the host calls' table layout (csrc/host_tables.h): the tables of a call do
// not overlap, are aligned, end within the context's block, and the copy holds the call's
// records and at most 15 bytes between them, whatever the context's capacity.
#include <stdint.h>
#include <stdio.h>

#include "ctm.h"
#include "host_tables.h"

#define CHECK(c)                                                  \
    do {                                                          \
        if (!(c)) {                                               \
            fprintf(stderr, "FAIL line %d: %s\n", __LINE__, #c); \
            return 1;                                             \
        }                                                         \
    } while (0)

int main()
{
    const size_t F = sizeof(ctm_frame), X = sizeof(ctm_box);
    const size_t frames[] = {1, 2, 3, 31, 32, 16383}, boxes[] = {0, 1, 2, 5, 63, 1 << 22};
    for (size_t cf : frames)
        for (size_t cb : boxes) {
            const ctm::HostTables cap = ctm::host_tables(cf, cf, cb, F, X);
            for (size_t n : frames)
                for (size_t b : boxes)
                    for (int mapped = 0; mapped < 2; ++mapped) {
                        if (n > cf || b > cb) continue;
                        const ctm::HostTables t = ctm::host_tables(n, mapped ? n : 0, b, F, X);
                        CHECK(t.frames >= ctm::kHostCountsBytes && t.frames % alignof(ctm_frame) == 0);
                        CHECK(t.sources >= t.frames + n * F && t.sources % alignof(ctm_frame) == 0);
                        CHECK(t.boxes >= t.sources + (mapped ? n * F : 0) && t.boxes % alignof(ctm_box) == 0);
                        CHECK(t.bytes >= t.boxes + b * X && t.bytes <= cap.bytes);
                        CHECK(t.bytes <= ctm::kHostCountsBytes + (mapped ? 2 : 1) * n * F + b * X + 15);
                    }
        }
    printf("OK\n");
    return 0;
}
