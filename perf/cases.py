"""Performance cases of the library: the calls a user of it makes, with their sizes.

Five operations, each through the public Python entry points:

- ``product``: ``sqnn_decode_matmul``, one layer of a model being served.  Batch 1 to 15 is token-by-token
  serving of a few requests (activations fp32 or bf16), batch 16 and more is a prompt, a larger serving
  batch or the image patches of a convolution (activations bf16);
- ``bits``: ``sqnn_decode`` to packed bit-planes, for users that consume the planes themselves;
- ``bf16``: ``sqnn_decode`` to a dense bf16 matrix, for users that hand the weights to another library;
- ``encode``: ``sqnn_encode_host``, Algorithm 1 over a quantized layer in host memory;
- ``search``: ``sqnn_search_seeds``, the exhaustive search for the best seeds on the device.

Layers are synthetic: normal weights, magnitude pruning over the layer, greedy binary codes per row, a
random XOR network per seed.  Where a layer has very many weights its planes and mask are drawn directly
(equiprobable bits, independent pruning).
"""
import numpy as np
import torch

from paper_1905_10138_b200 import sqnn
from paper_1905_10138_b200 import workloads as wl

DIRECT_ABOVE = 1 << 27          # weights per plane from which planes and mask are drawn as bits

# networks with compile-time kernels, and others a user may pick (odd, wide and small shapes)
NETS = ((40, 12), (40, 16), (60, 12), (80, 8), (80, 16), (100, 10), (200, 10))
OTHER_NETS = ((200, 20), (96, 14), (64, 16), (50, 20), (33, 20), (128, 24), (13, 5))


def _case(name, op, m, n, n_q, net, prune, batch=0, x="none"):
    c = {"op": op, "m": m, "n": n, "n_q": n_q, "n_out": net[0], "n_in": net[1], "prune": prune, "batch": batch, "x": x}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest layer of the configurations: all launch and latency
        _case("product_tiny_b1", "product", 256, 256, 1, (80, 8), 0.90, 1, "f32"),
        # AlexNet FC6, one activation vector: the benchmark's headline step
        _case("product_fc6_b1", "product", 4096, 9216, 1, (100, 10), 0.91, 1, "bf16"),
        # the gates of an LSTM, two bit-planes, eight requests at once
        _case("product_lstm_b8", "product", 6000, 3000, 2, (60, 12), 0.80, 8, "bf16"),
        # a layer with odd sizes and a network of the user's own, fp32 activations, four requests
        _case("product_odd_f32_b4", "product", 3001, 4099, 2, (96, 14), 0.85, 4, "f32"),
        # the LSTM gates over a batch: rows that do not start on word boundaries
        _case("product_lstm_b32", "product", 6000, 3000, 2, (60, 12), 0.80, 32, "bf16"),
        # AlexNet FC6 over a batch
        _case("product_fc6_b64", "product", 4096, 9216, 1, (100, 10), 0.91, 64, "bf16"),
        # a transformer's feed-forward matrix, three bit-planes, a prompt of 512 tokens
        _case("product_ffn_b512", "product", 4096, 16384, 3, (40, 12), 0.70, 512, "bf16"),
        # decode-only, one plane of 2^30 weights: the largest size of the configurations
        _case("bits_2p30", "bits", 32768, 32768, 1, (100, 10), 0.90),
        # planes of a layer with odd sizes and a network of the user's own
        _case("bits_odd", "bits", 5003, 7001, 2, (200, 20), 0.90),
        # the feed-forward matrix as a dense bf16 matrix
        _case("bf16_ffn", "bf16", 4096, 16384, 3, (40, 12), 0.70),
        # encoding of AlexNet FC6 (done once per layer and network)
        _case("encode_fc6", "encode", 4096, 9216, 1, (100, 10), 0.91),
        # the best seeds for the LSTM gates
        _case("search_lstm", "search", 6000, 3000, 2, (60, 12), 0.80),
    ]


def _log_size(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def draw(rng):
    """A layer of any size between the smallest and the largest listed ones of its operation."""
    op = rng.choice(("product",) * 7 + ("bits",) * 2 + ("bf16", "encode", "search"))
    net = rng.choice(NETS if rng.random() < 0.7 else OTHER_NETS)
    if op == "search" and net[1] > 16:
        net = rng.choice(NETS)
    # a network is chosen for its layer's density: about as many unpruned weights per slice as seed bits
    care = net[1] * rng.uniform(0.7, 1.3)
    prune = round(min(0.97, max(0.2, 1.0 - care / net[0])), 3)
    n_q = 1 if net[0] >= 80 and rng.random() < 0.7 else rng.choice((1, 2, 3))
    batch, x = 0, "none"
    top = {"product": 1 << 26, "bits": 1 << 28, "bf16": 1 << 27, "encode": 1 << 25, "search": 1 << 24}[op]
    if op == "search":                      # 2^n_in seeds per slice
        top = int(min(top, 2.4e9 / n_q / (1 << net[1]) * net[0]))
    weights = _log_size(rng, 1 << 16, max(1 << 16, top / n_q if op in ("bits", "bf16", "encode") else top))
    if op == "product":
        if rng.random() < 0.6:
            batch, x = rng.randint(1, 15) if rng.random() < 0.6 else 1, rng.choice(("bf16", "bf16", "f32"))
        else:
            batch, x = int(_log_size(rng, 16, 512)), "bf16"
    n = int(min(16384, max(64, weights ** 0.5 * _log_size(rng, 0.4, 2.5))))
    m = max(16, int(weights / n))
    if rng.random() < 0.6:                  # most layers have sizes that are multiples of a power of two
        m, n = max(64, m // 64 * 64), max(64, n // 64 * 64)
    return _case("", op, m, n, n_q, net, prune, batch, x)


def _pack(bits):
    """A CUDA tensor of booleans (flat) as packed 64-bit words, bit p of the vector = bit p % 64 of word p // 64."""
    pad = -bits.numel() % 64
    if pad:
        bits = torch.cat([bits, bits.new_zeros(pad)])
    weight = torch.tensor([1, 2, 4, 8, 16, 32, 64, 128], dtype=torch.uint8, device="cuda")
    return (bits.view(-1, 8).to(torch.uint8) * weight).sum(1, dtype=torch.uint8).view(torch.int64)


def _layer(case, g):
    """Packed planes (n_q vectors), packed mask and scales of a layer, on the GPU."""
    m, n, n_q = case["m"], case["n"], case["n_q"]
    mn = m * n
    if mn > DIRECT_ABOVE:
        words = (mn + 63) // 64
        planes = torch.randint(-(1 << 63), (1 << 63) - 1, (n_q * words,), dtype=torch.int64, device="cuda", generator=g)
        chunk = 1 << 26
        mask = torch.cat([_pack(torch.rand(min(chunk, mn - a), device="cuda", generator=g) >= case["prune"])
                          for a in range(0, mn, chunk)])
        return planes, mask, torch.rand((m, n_q), device="cuda", generator=g) + 0.5
    w = torch.randn((m, n), device="cuda", generator=g) * 0.02
    keep = max(1, round((1.0 - case["prune"]) * mn))
    mask = w.abs() >= torch.kthvalue(w.abs().flatten(), mn - keep + 1).values
    count = mask.sum(1, keepdim=True).clamp(min=1)
    planes, alpha = [], []
    for _ in range(n_q):
        b = w >= 0
        a = torch.where(mask, w.abs(), 0.0).sum(1, keepdim=True) / count
        planes.append(_pack(b.flatten()))
        alpha.append(a)
        w = w - torch.where(b, a, -a)
    return torch.cat(planes), _pack(mask.flatten()), torch.cat(alpha, 1).contiguous()


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    m, n, n_q, op, batch = case["m"], case["n"], case["n_q"], case["op"], case["batch"]
    rows = wl.network_rows(wl.xor_network(case["n_out"], case["n_in"], seed))
    planes, mask, alpha = _layer(case, g)
    s = {"op": op, "rows": rows, "n_in": case["n_in"], "m": m, "n": n, "n_q": n_q}
    if op == "search":
        slices = (m * n + case["n_out"] - 1) // case["n_out"]
        return dict(s, planes=planes, mask=mask, wc=torch.zeros(n_q * slices, dtype=torch.int32, device="cuda"),
                    np=torch.zeros(n_q * slices, dtype=torch.int16, device="cuda"))
    h_planes, h_mask = planes.cpu().numpy().view(np.uint64), mask.cpu().numpy().view(np.uint64)
    if op == "encode":
        # the blob goes into a staging buffer of fixed capacity (its size depends on the number of patches),
        # from which it would be written out or uploaded
        slices = m * n // case["n_out"] + 1024
        room = (1 << 16) + n_q * (slices * case["n_in"] // 8 + slices // 64 + 2 * int(mask.numel() * 64 * (1.0 - case["prune"]) * 1.02))
        return dict(s, planes=h_planes, mask=h_mask, staging=np.zeros(room, dtype=np.uint8))
    blob, _ = sqnn.sqnn_encode_host(rows, case["n_in"], m, n, n_q, h_planes, h_mask)
    s.update(desc=sqnn.sqnn_describe_host(blob), blob=torch.from_numpy(blob).cuda(), mask=mask, alpha=alpha,
             status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    if op == "bits":
        s["out"] = torch.empty(n_q * ((m * n + 63) // 64), dtype=torch.int64, device="cuda")
    elif op == "bf16":
        s["out"] = torch.empty((m, n), dtype=torch.bfloat16, device="cuda")
    else:
        dtype = torch.float32 if case["x"] == "f32" else torch.bfloat16
        pitch = (n + 7) // 8 * 8                # rows of a batch start on 16-byte boundaries
        x = torch.randn((batch, pitch), device="cuda", generator=g).to(dtype)
        s["x"] = x[:, :n]
        s["y"] = torch.empty((batch, m), dtype=torch.float32, device="cuda")
        need = sqnn.sqnn_workspace_bytes(s["desc"], batch)
        s["ws"] = torch.empty(need, dtype=torch.uint8, device="cuda") if need else None
    return s


def run(s):
    op = s["op"]
    if op == "product":
        sqnn.sqnn_decode_matmul(s["desc"], s["blob"], s["mask"], s["alpha"], s["x"], s["y"], s["ws"], s["status"])
        return s["y"]
    if op == "bits":
        sqnn.sqnn_decode(s["desc"], s["blob"], None, None, sqnn.OUT_BITS, s["out"], s["status"])
        return s["out"]
    if op == "bf16":
        sqnn.sqnn_decode(s["desc"], s["blob"], s["mask"], s["alpha"], sqnn.OUT_BF16, s["out"], s["status"])
        return s["out"]
    if op == "search":
        sqnn.sqnn_search_seeds(s["rows"], s["n_in"], s["m"], s["n"], s["n_q"], s["planes"], s["mask"], s["wc"], s["np"])
        return {"wc": s["wc"], "np": s["np"]}
    blob, stats = sqnn.sqnn_encode_host(s["rows"], s["n_in"], s["m"], s["n"], s["n_q"], s["planes"], s["mask"])
    s["staging"][:blob.size] = blob
    return {"blob": s["staging"], "bytes": blob.size, "stats": stats}


def work(case):
    """Bytes: compressed planes (n_in bits per slice; patches, a few per cent on top, are not counted), mask
    and scales where the operation reads them, activations and outputs.  flops: of the product, a multiply-add
    per unpruned weight and activation vector and the sum of a weight's scales; of a search or an encoding, one
    operation per unpruned weight and seed bit."""
    m, n, n_q, op, batch = case["m"], case["n"], case["n_q"], case["op"], case["batch"]
    mn = m * n
    stream = mn * n_q * case["n_in"] / case["n_out"] / 8
    kept = (1.0 - case["prune"]) * mn
    if op == "product":
        return {"bytes": stream + mn / 8 + 4 * m * n_q + batch * n * (4 if case["x"] == "f32" else 2) + 4 * batch * m,
                "flops": kept * (n_q + 2 * batch)}
    if op == "bits":
        return {"bytes": stream + mn * n_q / 8, "flops": 0}
    if op == "bf16":
        return {"bytes": stream + mn / 8 + 4 * m * n_q + 2 * mn, "flops": kept * n_q}
    if op == "encode":
        return {"bytes": mn * (n_q + 1) / 8 + stream, "flops": kept * n_q * case["n_in"]}
    slices = (mn + case["n_out"] - 1) // case["n_out"]
    return {"bytes": mn * (n_q + 1) / 8 + 6 * slices * n_q, "flops": kept * n_q * case["n_in"]}


def tolerance(case):
    """Bits, bytes and seeds are exact; a bf16 weight is one correctly rounded value.  Products are fp32 sums of
    exact terms whose order is free: short ones (plain sums) and long ones (tensor-core accumulation)."""
    if case["op"] != "product":
        return "exact"
    return {"rel": 1e-5 if case["batch"] <= 15 else 2e-5}
