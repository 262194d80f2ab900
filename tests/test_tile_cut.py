"""Kernel tiles of run-time network shapes: which layers the rule (cut_tiles) decodes in parts of format tiles and in how many turns of
32 slices a part, and the kernels on both sides of the line at layers of the size where a user meets them."""
import os
import subprocess

import numpy as np
import pytest

from oracle import oracle as orc
from paper_1905_10138_b200 import sqnn
from paper_1905_10138_b200 import workloads as wl
from tests import helpers as H
from tests.test_gpu_decode import generic_layer

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS, DECODE_WARPS = 148, 24

# Parts: (n_out, n_in, m, n, keep, n_q) and the turns of planes (by themselves and as the first half of a product), bf16 weights and the two forms of
# the small-batch product (0: whole format tiles).  Two to ten turns (the words of the slice that crosses from one turn into the next, seeds requested
# again after four turns, parts longer than a format tile, which take patch runs of three), for slices of 33 to 64, 65 to 128 and more bits.
PARTS = [
    ((33, 20, 2100, 5208, 0.7, 3), (10, 10, 4, 0, 0)),
    ((33, 7, 5500, 5000, 0.25, 1), (0, 0, 8, 10, 10)),
    ((50, 20, 2300, 5003, 0.3, 2), (5, 5, 3, 0, 0)),
    ((65, 10, 6000, 5001, 0.2, 1), (7, 5, 5, 6, 6)),
    ((129, 8, 4600, 5000, 0.1, 2), (5, 4, 2, 5, 5)),
]
# Whole format tiles: slices of no whole words of every table width and of 1, 2, 4, 5, 7 and 8 whole words, one to three planes, columns
# that are and are not a multiple of 32.
WHOLE = [
    (13, 5, 3700, 4001, 0.4, 1), (24, 6, 1900, 2003, 0.3, 2), (32, 9, 1900, 2016, 0.3, 2), (36, 8, 2500, 3001, 0.25, 3), (64, 11, 1900, 4000, 0.2, 2),
    (68, 10, 3700, 4001, 0.2, 2), (128, 24, 3700, 4000, 0.2, 2), (132, 8, 5600, 5301, 0.08, 1), (160, 20, 4300, 4301, 0.12, 1),
    (224, 32, 6400, 4001, 0.15, 1), (256, 32, 7300, 4000, 0.15, 1),
]
ids = [f"{c[0]}x{c[1]}-{c[2]}x{c[3]}-q{c[5]}" for c in [p for p, _ in PARTS] + WHOLE]

HARNESS = r"""
#include "sqnn_gemv_plan.h"
#include "sqnn_layout.h"
#include <cstdio>
#include <initializer_list>
using namespace sqnn;
int main()
{
    unsigned n_out, n_in, n_q, sms, decode_warps;
    unsigned long long m, n;
    while (std::scanf("%u %u %llu %llu %u %u %u", &n_out, &n_in, &m, &n, &n_q, &sms, &decode_warps) == 7) {
        const unsigned whole = format_tiles_per_kernel_tile(n_out), whole_words = 8 * whole * n_out / 32;
        for (DecodeFor what : {DecodeFor::PLANES, DecodeFor::PRODUCT, DecodeFor::BF16}) {
            unsigned KT = whole, W = whole_words;
            const unsigned turns = cut_decode_tiles(what, n_out, n_in, (m * n + 63) / 64, what == DecodeFor::BF16 ? 1 : n_q, sms, decode_warps, &KT, &W);
            std::printf("%u %u %u ", turns, KT, W);
        }
        GemvLayer L;
        L.m = m; L.n = n; L.n_q = n_q; L.sms = sms; L.W = whole_words;
        L.batch = 1; L.x_bytes = 2; L.tab_words = table_words(n_out, n_in); L.density = 0.1;
        const GemvForms f = plan_run_time_shape(n_out, n_in, L);
        for (const GemvTiles &t : {f.tc_tiles, f.walk_tiles}) {
            unsigned turns = 0;
            for (unsigned k = 1; t.KT == 0 && turns == 0; ++k) if (range_words(n_out, k) == t.W) turns = k;
            std::printf("%u %u %u ", turns, t.KT, t.W);
        }
        // whether a row fits: the two forms with whole tiles, and as cut
        std::printf("%u %u %u %u ", plan_gemv_tc(L).ok, f.tc.ok, plan_walk(L).ok, f.walk.ok);
        for (unsigned turns = 1; turns <= 10; ++turns) std::printf("%u ", range_words(n_out, turns));
        std::printf("\n");
    }
}
"""


@pytest.fixture(scope="module")
def cuts(tmp_path_factory):
    d = tmp_path_factory.mktemp("cut")
    src, exe = str(d / "cut.cpp"), str(d / "cut")
    with open(src, "w") as f:
        f.write(HARNESS)
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-I", os.path.join(ROOT, "paper_1905_10138_b200", "csrc"), src, "-o", exe], check=True)

    def run(layers):
        text = "\n".join(f"{n_out} {n_in} {m} {n} {n_q} {SMS} {DECODE_WARPS}" for n_out, n_in, m, n, _, n_q in layers)
        rows = [[int(x) for x in line.split()] for line in subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.splitlines()]
        return [([tuple(r[3 * i:3 * i + 3]) for i in range(5)], r[19:], r[15:19]) for r in rows]
    return run


def test_the_layers_below_are_cut_as_they_are_meant_to_be(cuts):
    for (case, turns), (got, words, _) in zip(PARTS, cuts([c for c, _ in PARTS])):
        for want, (t, kt, w) in zip(turns, got):
            assert t == want and (kt == 0) == (want > 0) and (want == 0 or w == words[want - 1]), (case, turns, got)
    for case, (got, *_) in zip(WHOLE, cuts(WHOLE)):
        assert all(kt != 0 for _, kt, _ in got), (case, got)


# (n_out, n_in, m, n, keep, n_q), what (as above), turns: calls that were timed in parts and in whole tiles.  Those without a turn took up to 1.34 of
# the time when they were cut.
TIMED = [
    ((24, 7, 1728, 640, 0.3, 3), 0, 0), ((44, 3, 3008, 2048, 0.05, 1), 0, 0), ((56, 5, 1344, 2560, 0.1, 1), 0, 0), ((112, 20, 3840, 3008, 0.2, 1), 0, 0),
    ((112, 10, 2000, 1200, 0.1, 2), 1, 0), ((64, 8, 3200, 768, 0.1, 3), 1, 0), ((112, 3, 7351, 1872, 0.02, 1), 3, 0), ((50, 5, 3008, 5184, 0.1, 1), 3, 0),
    ((8, 2, 960, 576, 0.2, 1), 4, 0), ((256, 4, 8000, 1984, 0.01, 1), 4, 0), ((40, 8, 4736, 768, 0.1, 1), 4, 0),
    ((50, 9, 3390, 870, 0.2, 1), 0, 2), ((240, 16, 2752, 4480, 0.05, 2), 0, 2), ((33, 20, 3648, 3072, 0.5, 3), 0, 10), ((128, 24, 1984, 1152, 0.2, 1), 3, 1),
    ((96, 7, 2880, 2048, 0.1, 1), 3, 1), ((127, 12, 1046, 944, 0.1, 1), 4, 1),
]


def test_calls_that_whole_tiles_take_less_time_for_are_not_cut(cuts):
    for (case, what, turns), (got, *_) in zip(TIMED, cuts([c for c, _, _ in TIMED])):
        assert got[what][0] == turns, (case, what, turns, got)


def test_rows_that_fit_in_parts_only_get_them_whatever_whole_tiles_would_cost(cuts):
    """Eight planes of 254-bit slices: two whole tiles (16 KB each) of every plane and the mask do not fit an SM's shared memory."""
    [(got, _, (tc_whole, tc, walk_whole, walk))] = cuts([(254, 8, 100, 20000, 0.05, 8)])
    assert (tc_whole, tc, walk_whole, walk) == (0, 1, 0, 1)
    assert got[3][1] == got[4][1] == 0


def test_a_part_of_t_turns_overlaps_no_more_than_32_t_slices(cuts):
    """Wherever it starts.  (One word per lane is the least, so slices of less than 33 bits may need more than one turn for it.)"""
    layers = [(n_out, 1, 100, 100, 0.1, 1) for n_out in range(1, 257)]
    for (n_out, *_), (_, words, _) in zip(layers, cuts(layers)):
        for turns in range(1, 11):
            w = words[turns - 1]
            if w == 1 and 1024 > (32 * turns - 1) * n_out:
                continue
            starts = {0} if n_out % 32 == 0 else range(n_out)             # bits of the first slice that lie before the part
            assert max(-(-(1024 * w + s) // n_out) for s in starts) <= 32 * turns, (n_out, turns)


def check(layer, bf16=True, products=((1, "bfloat16"), (3, "float32"), (16, "bfloat16"))):
    import torch
    blob, _ = H.blob_from_library(layer)
    dev = H.DeviceLayer(layer, blob)
    ref = np.empty((layer.n_q, layer.m, layer.n), dtype=np.uint8)
    got = dev.decode_bits()
    for i in range(layer.n_q):
        wc, np_, dp = sqnn.sqnn_unpack_host(blob, i)
        bits = orc.decode_plane(layer.M, layer.mn, wc.astype(np.uint64), np_, dp)
        assert np.array_equal(got[i], wl.pack_bits(bits)), i
        ref[i] = bits.reshape(layer.m, layer.n)
    if bf16:
        _, want = orc.reconstruct(ref, layer.mask, layer.alpha, want_f32=False)
        assert np.array_equal(dev.decode_bf16(), want)
    for batch, dtype in products:
        if batch > 15 and layer.n % 8:                               # a batch needs rows on 16-byte boundaries
            continue
        dtype = getattr(torch, dtype)
        x = torch.randn((batch, layer.n), generator=torch.Generator().manual_seed(batch)).to(dtype).float().numpy()
        # weights and activations enter exactly: what is left are fp32 sums, whose tolerance is the reading taken for all products
        assert H.rel_err(dev.matmul(x, dtype), orc.matmul(ref, layer.mask, layer.alpha, x.astype(np.float64))) <= 1e-4
    assert dev.status_value() == 0


@pytest.mark.gpu
@pytest.mark.parametrize("case", [p for p, _ in PARTS] + WHOLE, ids=ids)
def test_run_time_shapes_in_parts_of_many_turns_and_in_whole_tiles(case):
    n_out, n_in, m, n, keep, n_q = case
    check(generic_layer(n_out, n_in, m, n, keep, 80 + n_out, n_q=n_q))


@pytest.mark.gpu
def test_small_batch_product_of_rows_that_fit_in_parts_only():
    import torch
    layer = generic_layer(254, 8, 3, 20000, 0.05, 79, n_q=8)
    ref = H.oracle_decode(layer, H.oracle_encode(layer))
    dev = H.DeviceLayer(layer, H.blob_from_library(layer)[0])
    for batch, dtype in ((1, torch.bfloat16), (2, torch.float32)):
        x = torch.randn((batch, layer.n), generator=torch.Generator().manual_seed(batch)).to(dtype).float().numpy()
        assert H.rel_err(dev.matmul(x, dtype), orc.matmul(ref, layer.mask, layer.alpha, x.astype(np.float64))) <= 1e-4
    assert dev.status_value() == 0


# bf16 weights of the shapes with compile-time kernels: in parts (the first), and with more than four format tiles per SM, where their own kernels
# run: columns that are and are not a multiple of 32, rows on either side of the length from which on lanes that straddle rows take the plain
# way, one to four planes, scales whose sums vanish or are tiny.
COMPILED = [(40, 12, 1000, 5000, 1), (40, 12, 1600, 4000, 4), (40, 12, 1600, 4000, 3), (60, 12, 2300, 4099, 2), (80, 8, 3100, 4000, 1), (100, 10, 3900, 4001, 1),
            (100, 10, 2500, 6143, 2), (40, 12, 1000, 6145, 3), (60, 12, 1400, 7001, 2), (100, 10, 900, 17003, 1), (200, 10, 4400, 7003, 1)]


@pytest.mark.gpu
@pytest.mark.parametrize("n_out,n_in,m,n,n_q", COMPILED, ids=[f"{a}x{b}-{c}x{d}-q{q}" for a, b, c, d, q in COMPILED])
def test_bf16_weights_of_compile_time_shapes_with_odd_scales(n_out, n_in, m, n, n_q):
    layer = generic_layer(n_out, n_in, m, n, 0.3, 90 + n_q, n_q=n_q)
    layer.alpha[1::5] = 0.0
    layer.alpha[2::5] = 1e-38
    layer.alpha[3::5] = layer.alpha[3::5, :1]                 # sums that cancel
    layer.alpha[4::5, 0] = -1.5
    check(layer, products=())
