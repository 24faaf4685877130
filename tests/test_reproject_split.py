"""How a silhouette call is split over CTAs (reproject_split), checked on the
CPU: the bands cover the image, and calls of few masks with long lists get the
CTAs that keep the GPU busy instead of a cluster per mask."""

import os
import subprocess

import pytest

from paper_1311_6811_gb300 import build as libbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS = 152
BAND = 216 * 1024 * 8


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    libbuild.build()
    d = tmp_path_factory.mktemp("split")
    out = d / "reproject_split"
    objs = [os.path.join(libbuild.BUILD, f) for f in sorted(os.listdir(libbuild.BUILD)) if f.endswith(".o")]
    subprocess.run([libbuild.nvcc(), *libbuild.ARCH, "-std=c++17", "-I", os.path.join(ROOT, "include"),
                    "-I", libbuild.CSRC, os.path.join(ROOT, "tests", "host", "reproject_split.cu"), *objs,
                    "-o", str(out)], check=True, capture_output=True)

    def run(calls):
        inp = d / "calls.txt"
        inp.write_text("".join("%d %d %d %d\n" % c for c in calls))
        lines = subprocess.run([str(out), str(inp)], capture_output=True, text=True, check=True).stdout.splitlines()
        return [tuple(map(int, l.split())) for l in lines]
    return run


def test_every_split_is_launchable(split):
    calls = [(n_pix, masks, stride, sms) for n_pix in (1, 33, 67 * 51, 640 * 480, BAND - 1, BAND, BAND + 1, 1280 * 720,
                                                       1920 * 1080, 3840 * 2160, 1 << 28)
             for masks in (1, 2, 7, 8, 19, 30, 31, 36, 38, 39, 50, 51, 100, 800, 65535 * 32)
             for stride in (0, 1, 127, 4096, 4097, 262144, 1 << 24, (1 << 32) - 1) for sms in (1, 76, SMS)]
    for (n_pix, masks, stride, sms), (bands, band_pix, cluster, threads, most, parts, part_threads) in zip(calls, split(calls)):
        assert band_pix % 32 == 0 and 0 < band_pix <= BAND, (n_pix, bands, band_pix)
        assert (bands - 1) * band_pix < n_pix <= bands * band_pix
        assert cluster in (1, 2, 4, 8) and threads in (512, 1024)
        # CTAs fit the SM: bitmask and static shared memory, 64 registers a thread
        assert band_pix // 8 + 8192 <= 232448 and (1024 // threads) * (band_pix // 8 + 8192) <= 233472
        if parts:
            assert most < stride and parts * masks * bands <= 4 * sms and (parts - 1) * 128 < stride
            assert part_threads % 32 == 0 and 256 <= part_threads <= 1024
            assert (1024 // part_threads) * (band_pix // 8 + 8192) <= 233472
        else:
            assert parts == 0 and most == (1 << 32) - 1   # the clusters take every list


def test_few_masks_with_long_lists_fill_the_gpu(split):
    """Nearly four CTAs per SM for the long lists of any few masks of 640 x
    480, however few; a cluster per mask is at most 8 CTAs."""
    calls = [(640 * 480, masks, 262144, SMS) for masks in range(1, 51)]
    for (_, masks, _, _), (_, _, _, _, most, parts, threads) in zip(calls, split(calls)):
        assert masks * parts > 3.5 * SMS and threads == 256 and most <= 4096, (masks, parts)
    # the bands of one large camera, one CTA per SM
    for n_pix, want in ((1280 * 720, 1), (1920 * 1080, 2), (3840 * 2160, 5)):
        (bands, _, _, _, _, parts, threads), = split([(n_pix, 1, 262144, SMS)])
        assert bands == want and bands * parts > 0.95 * SMS and threads == 1024


def test_many_masks_keep_their_clusters(split):
    for masks, want in ((64, (2, 4)), (72, (2, 4)), (128, (1, 2)), (160, (2, 4)), (320, (1, 2)), (800, (1,))):
        (_, _, cluster, _, _, parts, _), = split([(640 * 480, masks, 262144, SMS)])
        assert parts == 0 and cluster in want, (masks, cluster)
