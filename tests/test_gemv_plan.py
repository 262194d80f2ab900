"""Plans of the small-batch product (csrc/sqnn_gemv_plan.h, host code): everything a plan promises the kernels, over
random layers, and on which side of the line measured calls fall."""
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include "sqnn_gemv_plan.h"
#include "sqnn_layout.h"
#include <cstdio>
using namespace sqnn;
int main()
{
    unsigned long long m, n;
    unsigned batch, n_q, n_out, n_in, x_bytes;
    double patches;
    while (std::scanf("%llu %llu %u %u %u %u %u %lf", &m, &n, &n_q, &n_out, &n_in, &batch, &x_bytes, &patches) == 8) {
        GemvLayer L;
        L.m = m; L.n = n; L.batch = batch; L.n_q = n_q;
        L.W = 8 * format_tiles_per_kernel_tile(n_out) * n_out / 32;
        L.tab_words = table_words(n_out, n_in);
        L.x_bytes = x_bytes; L.sms = 148;
        L.density = care_density(n_out, n_in, patches);
        const TcPlan t = plan_gemv_tc(L);
        const WalkPlan w = plan_walk(L);
        std::printf("%u %u %u %u %u %u %u %u %u %u %zu %.6g  %u %u %u %u %u %u %u %u %u %u %zu %.6g  %d\n", t.ok, t.rows_per_block, t.rows_per_chunk,
                    t.grid, t.units, t.bt, t.N, t.region_words, t.alpha_words, t.part_words, t.smem, t.us, w.ok, w.rows_per_block, w.rows_per_chunk,
                    w.grid, w.warps, w.bt, w.parts, w.region_words, w.alpha_words, w.part_words + w.xs_words, w.smem, w.us, take_walk(L, t, w));
    }
}
"""
TC = "ok rpb rpc grid units bt N region alpha part smem us".split()
WALK = "ok rpb rpc grid warps bt parts region alpha part smem us".split()


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, exe = str(d / "plan.cpp"), str(d / "plan")
    with open(src, "w") as f:
        f.write(HARNESS)
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-I", os.path.join(ROOT, "paper_1905_10138_b200", "csrc"), src, "-o", exe], check=True)

    def run(layers):
        text = "\n".join(" ".join(map(str, l)) for l in layers)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.splitlines()
        assert len(out) == len(layers)
        res = []
        for line in out:
            v = [float(x) if "." in x or "e" in x else int(x) for x in line.split()]
            res.append((dict(zip(TC, v[:12])), dict(zip(WALK, v[12:24])), v[24]))
        return res
    return run


def test_plans_fit_and_cover_every_layer(plans):
    rng = random.Random(3)
    nets = [(40, 12), (60, 12), (80, 8), (100, 10), (200, 10), (13, 5), (33, 20), (50, 20), (128, 24), (256, 32), (1, 1)]
    layers = []
    for _ in range(3000):
        n_out, n_in = rng.choice(nets)
        m, n = int(2 ** rng.uniform(0, 17)), int(2 ** rng.uniform(0, 17))
        layers.append((m, n, rng.randint(1, 8), n_out, n_in, rng.randint(1, 15), rng.choice((2, 4)), round(rng.uniform(0, n_out / 3), 3)))
    refused = 0
    for (m, n, n_q, n_out, n_in, batch, xb, _), (t, w, walk) in zip(layers, plans(layers)):
        kt = 1 if n_out % 4 == 0 else 2 if n_out % 2 == 0 else 4
        tile_words = 32 * (8 * kt * n_out // 32)
        for p in (t, w):
            if not p["ok"]:
                continue
            assert p["us"] > 0 and p["smem"] <= 220 * 1024
            assert 1 <= p["rpc"] <= p["rpb"] and p["grid"] <= 148 and (p["grid"] - 1) * p["rpb"] < m <= p["grid"] * p["rpb"]
            assert p["alpha"] >= p["rpc"] * n_q
            for _ in range(4):                                   # chunks start at any row of a block
                ra = rng.randrange(m)
                rb = min(ra + p["rpc"], m)
                k0, k1 = ra * n // (32 * tile_words), -(-rb * n // (32 * tile_words))
                assert (k1 - k0) * tile_words <= p["region"]
                if p is t:                                       # the last bit a lane of the last row may read
                    o = (rb - 1) * n - k0 * 32 * tile_words + 8 * 128 * t["units"]
                    assert o + 256 <= 32 * t["region"]
        if t["ok"]:
            pieces = 3 if xb == 4 else 1
            assert 1024 * t["units"] >= n and t["units"] % 8 != 0
            assert 8 * t["bt"] * pieces <= t["N"] <= 96 and t["N"] % 16 == 0 and t["bt"] <= batch
            assert t["part"] >= 4 * t["rpc"] * t["bt"]
        if w["ok"]:
            assert w["part"] >= w["rpc"] * w["parts"] * w["bt"]
        assert walk == (w["ok"] and (not t["ok"] or (n_q == 1 and xb == 2 and w["us"] < 0.9 * t["us"])))
        refused += not t["ok"] and not w["ok"]
        if n * (n_q + 1) <= 1_300_000:
            assert t["ok"] or w["ok"]
    assert refused < 300


# (layer, 1 = walk): small and sparse calls that the walk does faster, calls that it does slower, and calls that stay with
# the expanding form for its smaller error
SIDES = [
    ((2048, 1024, 1, 100, 10, 1, 2, 0.1), 1),
    ((900, 700, 1, 200, 10, 4, 2, 0.1), 1),
    ((4096, 9216, 1, 100, 10, 1, 2, 0.5), 0),
    ((1024, 3072, 1, 100, 10, 4, 2, 0.5), 0),
    ((4096, 12288, 1, 100, 10, 4, 2, 0.5), 0),
    ((256, 256, 1, 80, 8, 1, 4, 0.6), 0),
    ((6000, 3000, 2, 60, 12, 1, 2, 1.0), 0),
    ((4096, 12288, 1, 100, 10, 4, 4, 0.5), 0),
    ((5, 100003, 1, 40, 12, 2, 2, 0.3), 1),                      # rows too long for the expanding form
    ((3, 50001, 1, 100, 10, 1, 4, 0.5), 1),
]


def test_both_sides_of_the_line(plans):
    for (layer, want), (t, w, walk) in zip(SIDES, plans([l for l, _ in SIDES])):
        assert walk == want, (layer, t["us"], w["us"])
