"""How the CTAs of a decode launch are dealt out to several shards (host code, compiled here alone)."""
from __future__ import annotations

import random
import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_2607_07046_gb300" / "csrc"
PROGRAM = r"""
#include "deal.h"
#include <cstdio>
int main() {
    int n, per, ctas, units[16], end[16];
    double bytes[16];
    while (scanf("%d %d %d", &n, &per, &ctas) == 3) {
        for (int s = 0; s < n; ++s) scanf("%d %lf", &units[s], &bytes[s]);
        printf("%d", vt::deal_ctas(bytes, units, per, n, ctas, end));
        for (int s = 0; s < n; ++s) printf(" %d", end[s]);
        printf("\n");
    }
}
"""


def test_ctas_dealt_to_shards(tmp_path):
    """No launch has more CTAs than it asks for, except where the shards' units need them; every shard
    has enough for its units and no more than one a unit; and where neither bound acts, a shard has
    its share by bytes to within one CTA."""
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    (tmp_path / "deal.cpp").write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-I", str(CSRC), str(tmp_path / "deal.cpp"), "-o", str(tmp_path / "deal")], check=True)
    rng = random.Random(5)
    cases = [(40, 296, [(3440, 3440), (3440, 3440), (4128, 4128)]), (40, 304, [(3096, 3096), (3096, 3096), (4816, 4816)]),
             (40, 148, [(1, 1)] * 16), (64, 152, [(5000, 5000)]), (40, 304, [(1, 1), (20000, 20000), (3, 3)])]
    for _ in range(3000):
        units = [max(1, int(2 ** rng.uniform(0, 14))) for _ in range(rng.randint(1, 16))]
        same = rng.random() < 0.5
        cases.append((rng.choice([4, 40, 64]), rng.choice([148, 152, 296, 304]),
                      [(u, u * (1 if same else rng.choice([1, 64, 4096]))) for u in units]))
    text = "".join(f"{len(sh)} {per} {ctas} " + " ".join(f"{u} {b}" for u, b in sh) + "\n" for per, ctas, sh in cases)
    out = subprocess.run([str(tmp_path / "deal")], input=text, capture_output=True, text=True, check=True).stdout
    for (per, ctas, shards), line in zip(cases, out.splitlines(), strict=True):
        total, *end = map(int, line.split())
        got = [b - a for a, b in zip([0] + end, end)]
        need = [-(-u // per) for u, _ in shards]
        assert total == end[-1]
        assert all(lo <= g <= u for lo, g, (u, _) in zip(need, got, shards)), (per, ctas, shards, got)
        assert total <= max(ctas, sum(need)), (per, ctas, shards, got)
        share = [ctas * b / sum(b for _, b in shards) for _, b in shards]
        if all(max(lo, 1) + 1 <= s <= u - 1 for lo, s, (u, _) in zip(need, share, shards)):
            assert all(abs(g - s) <= 1 for g, s in zip(got, share)), (per, ctas, shards, got)
