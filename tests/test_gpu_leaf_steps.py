"""The tcgen05 leaf kernel's short tiles, whose rows are stacked two or four times with the copies sharing each output piece's columns
out: buckets of 1 to 128 rows and more, numbers of K-blocks and pieces that do not divide by the copies, one piece only, pieces of 16
columns.  And the expansion of every 8-bit code."""
import numpy as np
import pytest
import torch

from oracle import fff_oracle as orc
from paper_2308_14711_b200 import workloads as wl
from tests import util

pytestmark = pytest.mark.gpu

C = wl.FFFConfig
CASES = [
    C("ls_l24", 384, 400, 9, 24, "gelu", "bf16", 24576, "normal"),           # 6 K-blocks, 4 pieces, the last of 16 columns
    C("ls_l32", 640, 1040, 9, 32, "relu", "bf16", 20000, "normal"),          # 10 K-blocks, 9 pieces, biases in the epilogue
    C("ls_l20_one_piece", 128, 16, 10, 20, "silu", "bf16", 40000, "normal"),  # 2 K-blocks, one piece
    C("ls_l40", 256, 272, 8, 40, "gelu_tanh", "bf16", 16000, "normal"),      # LP = 64
    C("ls_l64_clusters", 384, 656, 9, 64, "gelu", "bf16", 16384, "clusters"),
    C("ls_padded", 328, 528, 9, 18, "gelu", "bf16", 24576, "normal"),        # two operands of H
]


@pytest.mark.parametrize("cfg", CASES, ids=lambda c: c.name)
def test_short_tiles_match_the_oracle(cfg):
    case = util.make_case(cfg, seed=4)
    y_ref, leaf_ref = orc.forward_i(case.net, case.x, threads=util.ORACLE_THREADS)
    layer = util.make_layer(case)
    x = util.to_device(case.x, "bf16")
    layer.profile_begin(1)
    y, leaf = layer.forward_infer(x)
    torch.cuda.synchronize()
    assert [n for n, _ in layer.profile_end()[0]][-1] == "grouped_leaf_ff_umma" and layer.last_status() == 0
    np.testing.assert_array_equal(leaf.cpu().numpy(), leaf_ref)
    util.check_outputs(y, y_ref, "bf16")
    layer.close()


def codes_layer(cfg, w, c1, s1, c2, s2):
    from paper_2308_14711_b200.binding import FFFLayer
    dev = {k: util.to_device(w[k], "bf16") for k in ("node_w", "node_b", "b1", "b2")}
    put = lambda a: torch.from_numpy(a).cuda()
    return FFFLayer(cfg.D, cfg.O, cfg.depth, cfg.leaf_width, cfg.activation, "bf16", dev["node_w"], dev["node_b"], put(c1), dev["b1"],
                    put(c2), dev["b2"], w1_scale=put(s1), w2_scale=put(s2))


def decoded(codes, scale):
    v = torch.from_numpy(codes).view(torch.float8_e4m3fn).double().numpy()
    return v * scale.astype(np.float64).reshape(-1, 1, 1)


@pytest.mark.parametrize("l,nan", [(16, False), (32, False), (40, False), (32, True)])
@pytest.mark.parametrize("subnormal", [False, True])
def test_every_code_of_8_bit_weights(l, nan, subnormal):
    """All finite codes, or the subnormal ones alone (a layer of only those shows each of their bits); with a NaN code in one leaf's
    W2 every other output is unchanged."""
    cfg = C("codes", 256, 144, 3, l, "gelu", "bf16", 700, "normal")
    w = wl.make_weights(cfg, 5)
    rng = np.random.default_rng(l)
    codes = np.array([c for c in range(256) if (c & 0x7f) <= (0x07 if subnormal else 0x7e)], dtype=np.uint8)
    c1 = rng.choice(codes, size=w["w1"].shape).astype(np.uint8)
    c2 = rng.choice(codes, size=w["w2"].shape).astype(np.uint8)
    spread = [np.sqrt(np.mean(decoded(c, np.ones(len(c))) ** 2)) for c in (c1, c2)]        # sums of about 1
    s1 = (rng.uniform(0.5, 2, 8) / (spread[0] * np.sqrt(cfg.D))).astype(np.float32)
    s2 = (rng.uniform(0.5, 2, 8) / (spread[1] * np.sqrt(l))).astype(np.float32)
    net = orc.Net(cfg.D, cfg.O, cfg.depth, l, cfg.activation, w["node_w"], w["node_b"], decoded(c1, s1), w["b1"], decoded(c2, s2), w["b2"])
    src = wl.TokenSource(cfg, 5)
    wl.enforce_margin(src, lambda rows: orc.path_margin(net, rows, threads=util.ORACLE_THREADS))
    y_ref, leaf_ref = orc.forward_i(net, src.x, threads=util.ORACLE_THREADS)
    if nan:
        c2[3, 7, 5] = 0xff
    layer = codes_layer(cfg, w, c1, s1, c2, s2)
    y, leaf = layer.forward_infer(util.to_device(src.x, "bf16"))
    torch.cuda.synchronize()
    np.testing.assert_array_equal(leaf.cpu().numpy(), leaf_ref)
    bad = torch.zeros(y.shape, dtype=torch.bool)
    if nan:
        bad[torch.from_numpy(leaf_ref == 3), 7] = True
        assert bad.any()
    assert torch.equal(torch.isnan(y).cpu(), bad)
    util.check_outputs(torch.where(bad.cuda(), torch.zeros_like(y), y), np.where(bad.numpy(), 0.0, y_ref), "bf16")
    layer.close()
