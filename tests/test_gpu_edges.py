"""GPU parity at the edges of the kernels' tiles: remainders of rows, columns, batches and planes, the smallest
and largest sizes a dispatch hands to each form, values that need the plain way."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1905_10138_b200 import sqnn
from paper_1905_10138_b200 import workloads as wl
from tests import helpers as H
from tests.test_gpu_decode import generic_layer

pytestmark = pytest.mark.gpu


def product(layer, x, dtype):
    import torch
    ref_bits = H.oracle_decode(layer, H.oracle_encode(layer))
    ref = orc.matmul(ref_bits, layer.mask, layer.alpha, x.astype(np.float64))
    dev = H.DeviceLayer(layer, H.blob_from_library(layer)[0])
    y = dev.matmul(x, torch.float32 if dtype == "f32" else torch.bfloat16)
    assert dev.status_value() == 0
    return y, ref


# (n_out, n_in, m, n, keep, n_q, x, batch): one row; ranges of 128 columns with one column left over; 17 rows in
# the last tile of 16; the most vectors of one pass (12 bf16, 4 fp32) and one more; rows cut into chunks
SMALL = [
    (100, 10, 1, 1, 1.0, 1, "f32", 1),
    (100, 10, 17, 1025, 0.2, 1, "bf16", 12),
    (60, 12, 33, 1023, 0.2, 2, "bf16", 13),
    (40, 12, 149, 129, 0.3, 3, "f32", 4),
    (96, 14, 31, 2050, 0.15, 2, "f32", 5),
    (128, 24, 300, 640, 0.2, 8, "bf16", 15),
    (64, 16, 5000, 900, 0.25, 1, "f32", 3),
    (80, 16, 2500, 8192, 0.2, 3, "bf16", 2),
    # ranges of 2, 3, 4, 8 and 8 + 1 units of 128 columns: banks shared by none to all lanes of a row
    (60, 12, 40, 2048, 0.2, 2, "bf16", 8),
    (60, 12, 40, 2049, 0.2, 2, "bf16", 8),
    (100, 10, 200, 4096, 0.1, 1, "f32", 3),
    (100, 10, 33, 7169, 0.1, 1, "bf16", 5),
    (100, 10, 33, 8193, 0.1, 1, "bf16", 5),
]


@pytest.mark.parametrize("case", SMALL, ids=lambda c: "x".join(map(str, c)))
def test_small_batch_product_at_tile_edges(case):
    n_out, n_in, m, n, keep, n_q, x_dtype, batch = case
    layer = generic_layer(n_out, n_in, m, n, keep, 51, n_q=n_q)
    layer.x_dtype = x_dtype
    y, ref = product(layer, layer.activations(batch), x_dtype)
    assert H.rel_err(y, ref) <= 1e-4


# (n_out, n_in, m, n, keep, n_q, x, batch, walk): small and sparse one-plane bf16 layers go to the walk (one, two, four and
# eight vectors at a time, a row over several warps, chunks of rows, a second group of vectors), their neighbours do not
FORMS = [
    (100, 10, 300, 1024, 0.07, 1, "bf16", 1, True),
    (100, 10, 1, 64, 0.1, 1, "bf16", 1, True),
    (80, 8, 147, 3001, 0.1, 1, "bf16", 2, True),
    (200, 10, 900, 700, 0.03, 1, "bf16", 4, True),
    (200, 10, 149, 16384, 0.02, 1, "bf16", 15, False),
    (64, 16, 40, 44001, 0.25, 1, "f32", 11, True),              # (rows too long for the other form)
    (100, 10, 300, 1024, 0.07, 1, "f32", 1, False),
    (100, 10, 300, 1024, 0.07, 2, "bf16", 1, False),
    (60, 12, 2000, 3000, 0.2, 1, "bf16", 1, False),
]


@pytest.mark.parametrize("case", FORMS, ids=lambda c: "x".join(map(str, c)))
def test_small_batch_product_in_the_form_that_the_rule_picks(case):
    """Which form ran: with the library's test knob the tensor-core form hears of no completion and reports a timeout."""
    import torch
    n_out, n_in, m, n, keep, n_q, x_dtype, batch, walk = case
    layer = generic_layer(n_out, n_in, m, n, keep, 56, n_q=n_q)
    layer.x_dtype = x_dtype
    x = layer.activations(batch)
    y, ref = product(layer, x, x_dtype)
    assert H.rel_err(y, ref) <= 1e-4
    dev = H.DeviceLayer(layer, H.blob_from_library(layer)[0])
    try:
        sqnn.sqnn_set_debug_flags(2, 1_000_000)
        dev.matmul(x, torch.float32 if x_dtype == "f32" else torch.bfloat16)
    finally:
        sqnn.sqnn_set_debug_flags(0, 0)
    assert dev.status_value() == (0 if walk else -sqnn.E_TIMEOUT)


@pytest.mark.parametrize("x_dtype", ["f32", "bf16"])
def test_pruned_weights_do_not_meet_activations_that_are_not_finite(x_dtype):
    layer = generic_layer(100, 10, 40, 700, 0.3, 52)
    layer.x_dtype = x_dtype
    x = layer.activations(3)
    x[0, 5], x[1, 300], x[2, 699] = np.inf, np.nan, -np.inf
    y, _ = product(layer, np.where(np.isfinite(x), x, 0.0).astype(np.float32), x_dtype)
    dirty, _ = product(layer, x, x_dtype)
    for b, c in ((0, 5), (1, 300), (2, 699)):
        pruned = layer.mask[:, c] == 0
        assert np.allclose(dirty[b, pruned], y[b, pruned], rtol=1e-5, atol=1e-5)
        assert not np.isfinite(dirty[b, ~pruned]).any()


# batches around the tiles of the accumulators (1 to 4 units share 384 columns), planes in groups, a row more
# than a row tile, macros of 256 columns with 8 left over
LARGE = [
    (100, 10, 129, 264, 0.2, 1, 16),
    (100, 10, 257, 512, 0.2, 1, 193),
    (60, 12, 127, 1000, 0.2, 2, 97),
    (40, 12, 130, 768, 0.3, 3, 129),
    (96, 14, 40, 1032, 0.2, 4, 100),
    (64, 16, 140, 520, 0.25, 7, 33),
    (200, 10, 64, 8, 0.1, 1, 1024),
]


@pytest.mark.parametrize("case", LARGE, ids=lambda c: "x".join(map(str, c)))
def test_tensor_core_product_at_tile_edges(case):
    n_out, n_in, m, n, keep, n_q, batch = case
    layer = generic_layer(n_out, n_in, m, n, keep, 53, n_q=n_q)
    layer.x_dtype = "bf16"
    y, ref = product(layer, layer.activations(batch), "bf16")
    assert H.rel_err(y, ref) <= 2e-4


# The product's dynamic shared memory ends less than its static variables below 48 KB (49136, 49152, 48976 and 49008 bytes), where a
# launch needs a larger limit although the dynamic part alone does not.
JUST_BELOW_48_KB = [
    (100, 10, 18, 930, 0.1, 2, "f32", 2),
    (100, 10, 34, 1018, 0.1, 2, "bf16", 6),
    (96, 14, 47, 1031, 0.15, 2, "f32", 3),
    (64, 16, 56, 1049, 0.25, 3, "bf16", 10),
]


@pytest.mark.parametrize("case", JUST_BELOW_48_KB, ids=lambda c: "x".join(map(str, c)))
def test_small_batch_product_with_just_below_48_kb_of_shared_memory(case):
    n_out, n_in, m, n, keep, n_q, x_dtype, batch = case
    layer = generic_layer(n_out, n_in, m, n, keep, 57, n_q=n_q)
    layer.x_dtype = x_dtype
    y, ref = product(layer, layer.activations(batch), x_dtype)
    assert H.rel_err(y, ref) <= 1e-4


# n below, at and above the 8, 32 and 1024 columns at which a lane's words cross rows; whole-word and shifted
# run-time network shapes; scales whose sums vanish, are infinite or tiny
BF16 = [(40, 12, 50, 7, 2), (100, 10, 40, 33, 1), (60, 12, 9, 1024, 3), (60, 12, 9, 1025, 3), (200, 10, 30, 2001, 2),
        (96, 9, 20, 999, 3), (160, 20, 20, 999, 1), (33, 20, 31, 1500, 2), (224, 32, 16, 640, 2), (50, 20, 40, 801, 4)]


@pytest.mark.parametrize("n_out,n_in,m,n,n_q", BF16)
def test_bf16_weights_at_row_boundaries_and_with_odd_scales(n_out, n_in, m, n, n_q):
    layer = generic_layer(n_out, n_in, m, n, 0.3, 54, n_q=n_q)
    layer.alpha[1::5] = 0.0
    layer.alpha[2::5] = 1e-38
    layer.alpha[3::5] = layer.alpha[3::5, :1]                 # sums that cancel
    layer.alpha[4::5, 0] = -1.5
    arrays = H.oracle_encode(layer)
    ref_bits = H.oracle_decode(layer, arrays)
    dev = H.DeviceLayer(layer, H.blob_from_oracle(layer, arrays))
    got = dev.decode_bits()
    for i in range(n_q):
        assert np.array_equal(got[i], wl.pack_bits(ref_bits[i]))
    _, ref = orc.reconstruct(ref_bits, layer.mask, layer.alpha, want_f32=False)
    assert np.array_equal(dev.decode_bf16(), ref)


# more dependent rows than the candidate words hold, ranks above and below 12, rank-deficient networks
SEARCH = [(200, 8, 0.6, 1, False), (100, 14, 0.35, 2, False), (40, 16, 0.9, 1, False), (60, 12, 1.0, 1, True), (64, 17, 0.3, 1, False)]


@pytest.mark.parametrize("n_out,n_in,keep,n_q,deficient", SEARCH)
def test_seed_search_beyond_the_common_slices(n_out, n_in, keep, n_q, deficient):
    import torch
    layer = generic_layer(n_out, n_in, 3, 997 if n_in < 16 else 301, keep, 55, n_q=n_q)
    if deficient:
        layer.M[:, 3] = layer.M[:, 0] ^ layer.M[:, 1]
        layer.M[:, 7] = 0
    slices = (layer.mn + n_out - 1) // n_out
    planes = torch.from_numpy(np.concatenate([wl.pack_bits(layer.planes[i]) for i in range(n_q)]).view(np.int64)).cuda()
    mask = torch.from_numpy(wl.pack_bits(layer.mask).view(np.int64)).cuda()
    wc = torch.zeros(n_q * slices, dtype=torch.int32, device="cuda")
    np_ = torch.zeros(n_q * slices, dtype=torch.int16, device="cuda")
    sqnn.sqnn_search_seeds(wl.network_rows(layer.M), n_in, layer.m, layer.n, n_q, planes, mask, wc, np_)
    torch.cuda.synchronize()
    for i in range(n_q):
        owc, onp, _ = orc.encode_plane(layer.M, layer.planes[i].ravel(), layer.mask.ravel(), exhaustive=True)
        assert np.array_equal(wc.cpu().numpy().view(np.uint32)[i * slices:(i + 1) * slices].astype(np.uint64), owc)
        assert np.array_equal(np_.cpu().numpy()[i * slices:(i + 1) * slices], onp)
