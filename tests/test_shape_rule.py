"""The choice of a transform shape by batch size (csrc/shape_rule.h), compiled
as host code: every choice is a built shape, and clusters of more than 8 CTAs,
the portable size, are only taken where the GPU can place one."""
import os
import shutil
import subprocess

import pytest

from paper_2109_14704_gb300 import he
from paper_2109_14704_gb300.build import CSRC

PROGRAM = r"""
#include <stdio.h>
#include "shape_rule.h"
int main()
{
    unsigned log_n, items, inv, sms, wide;
    while (scanf("%u %u %u %u %u", &log_n, &items, &inv, &sms, &wide) == 5) {
        int s[4] = {0, 0, 0, 0};
        he::auto_shape((int)log_n, items, inv, sms, wide, s, s + 1);
        if (!inv) he::product_shape((int)log_n, items, sms, wide, s + 2, s + 3);
        printf("%d %d %d %d\n", s[0], s[1], s[2], s[3]);
    }
}
"""


@pytest.mark.parametrize("sms", [152, 148, 18])
def test_choices_are_built_and_portable_where_needed(tmp_path, sms):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("needs g++")
    (tmp_path / "p.cc").write_text(PROGRAM)
    exe = str(tmp_path / "p")
    subprocess.run([gxx, "-std=c++17", "-I", CSRC, str(tmp_path / "p.cc"), "-o", exe], check=True)
    edge = sorted({k for log_n in range(10, 17) for k in (sms * 4096 >> log_n, (sms * 4096 >> log_n) * 3 // 4)}
                  | {1, 8, sms // 8, sms // 4, 1 << 20})
    calls = [(log_n, items, inv, sms, wide) for log_n in range(10, 17)
             for items in sorted({e + d for e in edge for d in (-1, 0, 1)} - {0, -1}) for inv in (0, 1) for wide in (0, 1)]
    out = subprocess.run([exe], input="\n".join(" ".join(map(str, c)) for c in calls), check=True, text=True,
                         capture_output=True, env=dict(os.environ)).stdout.split("\n")
    for (log_n, items, inv, _, wide), line in zip(calls, out):
        shape, product = tuple(map(int, line.split()))[:2], tuple(map(int, line.split()))[2:]
        built = [s[:2] for s in he.ntt_shapes(1 << log_n) if not s[2]]
        for s in (shape, product):
            lb = s[0] or built[0][0]
            assert s == (0, 0) or s in built, (log_n, items, s)
            assert wide or (1 << log_n) >> lb <= 8, (log_n, items, s)
        if log_n == 13 and not inv and product == (11, 4):
            assert 4 * items <= sms - 8, items       # a CTA an SM, which clusters of four do not fill
        if log_n == 16:
            assert shape == ((12, 4) if wide else (0, 0))
