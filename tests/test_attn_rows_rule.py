"""Which separate attention kernel a step with a block of 17 to 128 rows takes (attn_rows_pays, compiled for
the host): the kernel that measured shorter, for steps of 32 heads on 152 SMs."""
import subprocess

import pytest

from paper_2609_26100_gb300 import build

PROGRAM = """
#include <cstdio>
#include <vector>
#include "internal.h"
int main() {
  int n;
  while (std::scanf("%d", &n) == 1) {
    std::vector<int> nodes(n), ctx(n);
    for (int b = 0; b < n; ++b)
      if (std::scanf("%d %d", &nodes[b], &ctx[b]) != 2) return 1;
    std::printf("%d\\n", tss::attn_rows_pays(n, [&](int b) { return (ctx[b] + nodes[b] + 63) / 64; },
                                            [&](int b) { return nodes[b]; }, 32, 152));
  }
}
"""
# (blocks, context of each): us a step of two 7B layers on attn_rows_kernel / the warp-level kernel
CASES = [
    ([17] * 8, 200, False),  # 542 / 523
    ([17] * 8, 4000, False),  # 944 / 843
    ([17] * 8, 16000, False),  # 2069 / 1714
    ([24] * 4, 16000, False),  # 1238 / 1196
    ([32] * 8, 1000, False),  # 792 / 763
    ([40] + [5] * 20, 4000, False),  # 1587 / 1253
    ([64] + [5] * 30, 1000, False),  # 1048 / 893
    ([64, 64] + [16] * 6, 12000, False),  # 1909 / 1611
    ([33] + [17] * 8, 12000, False),  # 1880 / 1664
    ([33] + [1] * 40, 1000, False),  # 922 / 698
    ([33, 1, 1], 12000, False),  # 865 / 725
    ([17], 2000, True),  # 323 / 329
    ([24], 16000, True),  # 524 / 543
    ([32] * 2, 8000, True),  # 565 / 599
    ([24] * 4, 4000, True),  # 601 / 619
    ([33], 1000, True),  # 340 / 373
    ([33] * 4, 16000, True),  # 1360 / 1594
    ([64] * 4, 1000, True),  # 723 / 804
    ([64], 16000, True),  # 572 / 715
    ([128] + [2] * 30, 4000, True),  # 2101 / 2414
    ([100] + [8] * 10, 1000, True),  # 759 / 786
]


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cu").write_text(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
                    str(d / "rule.cu"), "-o", str(d / "rule")], check=True)
    return str(d / "rule")


def test_rule_takes_the_shorter_kernel(rule):
    text = "\n".join(f"{len(blocks)} " + " ".join(f"{n} {ctx}" for n in blocks) for blocks, ctx, _ in CASES)
    got = subprocess.run([rule], input=text, check=True, capture_output=True, text=True).stdout.split()
    assert [x == "1" for x in got] == [rows for _, _, rows in CASES]
