// Host-only test driver: what the bounds-checked build tests of the adjoint's
// owner lists, for segments and entries read from a text file.
//
// input:  per line: e0 e1 base end total entry (an index into the lists)
// output: per line: whether the segment is in its slice, the entry in the slice
#include <cstdio>

#include "psfs_internal.cuh"

int main(int argc, char **argv)
{
    if (argc < 2) return 2;
    FILE *f = std::fopen(argv[1], "r");
    if (!f) return 2;
    static const uint32_t lists[1] = {0};   // only addresses are compared
    unsigned v[6];
    while (std::fscanf(f, "%u %u %u %u %u %u", &v[0], &v[1], &v[2], &v[3], &v[4], &v[5]) == 6)
        std::printf("%d %d\n", psfs::owner_segment_ok(v[0], v[1], v[2], v[3], v[4]) ? 1 : 0,
                    psfs::owner_entry_ok(lists + v[5], lists, v[2], v[3]) ? 1 : 0);
    std::fclose(f);
    return 0;
}
