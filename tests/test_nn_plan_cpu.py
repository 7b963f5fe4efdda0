"""The weight gradient's plan and its map from flat positions to pixels (csrc/nn_plan.cuh), compiled for the host and
walked position by position against plain 64-bit division: images far taller than a segment of the network's levels,
segments over several images, one and several column strips."""
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Walks at most `most` segments, spread over all of them, as the producers of conv3x3_wgrad do: the segment's positions
# and the ring's halo of one pitch on either side.
WALK = r"""
#include <cstdio>
#include <cstdlib>
#include "nn_plan.cuh"
using namespace lbm_nn;
int main(int argc, char** argv) {
  int v[6];
  for (int i = 0; i < 6; ++i) v[i] = atoi(argv[1 + i]);
  const int n = v[0], h = v[1], w = v[2], cin = v[3], cout = v[4], most = v[5];
  const WgradPlan p = wgrad_plan(n, h, w, cin, cout);
  long long nseg = 0, walked = 0, wrong = 0, far = 0;
  for (int pass = 0; pass < 2; ++pass) {
    const long long stride = nseg / most + 1;
    long long k = 0;
    for (long long z = 0; z < p.chunks; ++z) {
      const long long total = p.steps * p.strips, t0 = total * z / p.chunks, t1 = total * (z + 1) / p.chunks;
      for (long long t = t0, te; t < t1; t = te, ++k) {
        te = std::min(std::min(t1, t + p.seg_steps), (t / p.steps + 1) * p.steps);
        if (!pass || (k % stride && te < total)) continue;
        const int strip = (int)(t / p.steps), qb = (int)(te - t) * p.KP;
        const long long first = t % p.steps * p.KP;
        WgradSegment seg(p, h, w);
        seg.start(p, first, strip);
        for (int q = -p.pitch; q < qb + p.pitch; ++q) {
          if (q < seg.lo || q >= seg.hi) continue;
          int r, c;
          seg.map.split(q + seg.off, r, c);
          const unsigned rel = seg.map.offset(r, c);
          const long long got = rel == ~0u ? -1 : seg.map.origin() + rel;
          const long long at = first + q, row = at / p.pitch, img = row / (h + 1LL), yy = row % (h + 1LL),
                          xx = at % p.pitch + strip * p.Wt - 1;
          const long long want = yy < h && xx >= 0 && xx < w ? (img * h + yy) * w + xx : -1;
          ++walked;
          wrong += got != want;
          far = std::max(far, want);
        }
      }
    }
    nseg = k;
  }
  printf("%lld %lld %lld %lld %d %d\n", walked, wrong, far, nseg, p.slots, p.seg_steps * p.KP);
}
"""


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, exe = d / "walk.cpp", d / "walk"
    src.write_text(WALK)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2311_05091_gb300", "csrc"), "-x", "c++",
                    str(src), "-o", str(exe)], check=True)

    def run(n, h, w, cin, cout, most=16):
        out = subprocess.run([str(exe), *map(str, (n, h, w, cin, cout, most))], check=True, capture_output=True, text=True)
        return [int(k) for k in out.stdout.split()]   # walked, wrong, largest pixel, segments, slots, longest segment
    return run


# tall and narrow: a segment spans several images of tens of thousands of rows
@pytest.mark.parametrize("n,h,w,cin,cout", [(3, 65536, 1, 1024, 1024), (12, 65536, 1, 512, 512), (64, 65536, 2, 256, 256),
                                            (18, 55544, 4, 256, 256), (5, 46341, 1, 768, 768), (2, 200000, 3, 512, 1024),
                                            (300, 4000, 1, 256, 512), (16, 256, 256, 32, 32), (9, 1, 300, 48, 16),
                                            (3, 33, 32, 256, 144), (1000, 1, 1, 64, 64)])
def test_every_position_maps_to_its_pixel(walk, n, h, w, cin, cout):
    walked, wrong, *_ = walk(n, h, w, cin, cout)
    assert walked > 0 and wrong == 0


# 2^31 pixels and more: 128 GB a tensor of 16 channels, half of the device
@pytest.mark.parametrize("n,h,w", [(1, 65536, 40000), (3, 1 << 20, 1024), (40000, 256, 256), (1 << 20, 1, 2304),
                                   (1, (1 << 31) - 1, 1), (1, 1, (1 << 31) - 1), (2, (1 << 30) + 77, 1), (5, 3, 150000001)])
def test_pixels_beyond_32_bits(walk, n, h, w):
    walked, wrong, far, *_ = walk(n, h, w, 16, 16)
    assert walked > 0 and wrong == 0 and far == n * h * w - 1


def test_every_plan_has_a_slot_per_producer_group(walk):
    r = random.Random(11)
    for _ in range(300):
        n, h, w = r.randint(1, 20), r.randint(1, 300), r.choice([1, 2, 7, 31, 64, 127, 128, 129, 200, 256, 300, 1000])
        cin, cout = 16 * r.randint(1, 40), 16 * r.randint(1, 40)
        walked, wrong, far, segments, slots, longest = walk(n, h, w, cin, cout, 1)
        assert 3 <= slots <= 6 and segments >= 1 and longest >= 1 and wrong == 0, (n, h, w, cin, cout)
