// Host-only test driver: prints the split of silhouette calls over CTAs
// (reproject_split) for calls read from a text file, so that a test can check
// the rule without a GPU.
//
// input:  per call: n_pix frame_cams list_stride sms
// output: per call: bands band_pix cluster threads most parts part_threads
#include <cstdio>

#include "psfs_internal.cuh"

int main(int argc, char **argv)
{
    if (argc < 2) return 2;
    FILE *f = std::fopen(argv[1], "r");
    if (!f) return 2;
    long long n_pix = 0, frame_cams = 0;
    unsigned stride = 0;
    int sms = 0;
    while (std::fscanf(f, "%lld %lld %u %d", &n_pix, &frame_cams, &stride, &sms) == 4) {
        const psfs::ReprojectSplit r = psfs::reproject_split(n_pix, frame_cams, stride, sms);
        std::printf("%d %d %d %d %u %d %d\n", r.bands, r.band_pix, r.cluster, r.threads, r.most, r.parts,
                    r.part_threads);
    }
    std::fclose(f);
    return 0;
}
