"""The binning's division of work, host arithmetic of bin.cuh (no GPU needed): a
small program compiled against the header prints it for many frames."""

import os
import subprocess

import pytest

from paper_2410_04974_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "bin.cuh"
using namespace sixdgs;
int main() {
  long long n, tiles; int cams, sms;
  while (std::scanf("%lld %d %lld %d", &n, &cams, &tiles, &sms) == 4) {
    const ViewParts vp = view_parts(n, cams);
    const uint32_t segments = (uint32_t)((n + kStageTile - 1) / kStageTile) * vp.parts;
    const ScatterShare s = scatter_share(segments, (uint32_t)kStageTile * vp.views, (uint32_t)tiles, sms);
    std::printf("%u %u %u %u %u %u %d\n", vp.parts, vp.views, segments, s.grid, s.split, s.step,
                (int)defer_big_rects(n, cams, tiles));
  }
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cu").write_text(PROGRAM)
    subprocess.run([build.nvcc(), "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, *build.ARCH, str(d / "rules.cu"),
                    "-o", str(d / "rules")], check=True)

    def ask(frames):
        out = subprocess.run([str(d / "rules")], input="".join("%d %d %d %d\n" % f for f in frames), text=True,
                             capture_output=True, check=True, env=dict(os.environ)).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]

    return ask


def test_a_scatter_step_stays_within_32_bits_and_covers_its_segment(rules):
    frames = [(n, cams, tiles, sms) for n in (1, 127, 129, 5_000, 38_912, 200_000, 3_000_000) for cams in (1, 2, 7, 20, 256)
              for tiles in (1, 2_500, 1 << 20, 1 << 23, (1 << 24) + 3, 1 << 25, (1 << 31) - 1) for sms in (132, 152)]
    for (n, cams, tiles, sms), (parts, views, segments, grid, split, step, _) in zip(frames, rules(frames)):
        assert step >= 1 and step * tiles <= 1 << 31, (n, cams, tiles)     # prefix sums of a step: 32 bits
        size = 128 * views
        assert 1 <= split and 1 <= grid <= min(segments * split, 16 * sms)
        # CTA c of a segment's `split` takes [k step, (k + 1) step) for k = c, c + split, ...: every entry once
        assert split <= -(-size // step)
        # the views of every tile of Gaussians, each once
        assert (parts - 1) * views < cams <= parts * views and segments == -(-n // 128) * parts


@pytest.mark.parametrize("n,cams", [(1, 1), (1_000, 1), (2_000, 1), (200, 8)])
def test_few_pairs_are_scattered_by_a_cta_each(rules, n, cams):
    """Where each may touch tens of thousands of tiles."""
    (parts, views, segments, grid, split, step, _), = rules([(n, cams, 30_976 * cams, 152)])
    assert step == 1 and segments * 128 * views <= 16 * 152
    assert split == min(128 * views, 16 * 152 // segments) and grid == segments * split


def test_launch_count_of_a_step_follows_the_rule_for_large_rectangles(rules):
    import bench
    import synth
    from paper_2410_04974_gb300.render import make_plan, make_settings

    frames = [(n, cams, size) for n in (0, 1, 4_000, 17_133, 38_784, 38_785, 300_000) for cams in (1, 2, 3, 8, 20, 64)
              for size in (128, 512, 513, 1408)]
    plans = [make_plan(n, 3, synth.ring_cameras(cams, size, size), make_settings()) for n, cams, size in frames]
    asked = rules([(n, cams, int(p.total_tiles), 152) for (n, cams, _), p in zip(frames, plans)])
    seen = set()
    for (n, cams, size), plan, rule in zip(frames, plans, asked):
        count = n > 0 and bool(rule[6])
        # upload, projection, count, scan, scatter, sort, fused blend, per-Gaussian backward
        want = -(-cams // 48) + (n > 0) + count + 3 + 1 + (n > 0)
        assert bench.step_launches(plan) == want, (n, cams, size)
        seen.add(count)
    assert seen == {False, True}
