"""GPU parity: every C-ABI entry point against the fp64 oracle on the same seeded inputs.

Tolerances (rel-L2 = ||a-b||/||b||, b the oracle): merged weights and bias 1e-5 (fp32 FMA merge);
conv outputs 1e-4 in fp32 and 2e-2 in bf16 (bf16 rounding of the merged weights, of the input and
of the output; fp32 accumulation).  Every output is also held to the element-wise bound of
parity_util (a localised fault cannot hide under a whole-tensor norm), and every buffer the library
writes sits between sentinel bands that must come back untouched."""
import numpy as np
import pytest

from oracle import dc_oracle as O
from paper_2301_12187_b200 import inputs as I
from parity_util import Guarded, assert_close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL_W, TOL_F32, TOL_BF16 = 1e-5, 1e-4, 2e-2


@pytest.fixture(scope="module")
def dc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_12187_b200 import dc as _dc
    _dc.lib()
    return _dc


def dev(a, dtype=torch.float32):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype=dtype).contiguous()


def nchw(t):
    return t.float().cpu().numpy().astype(np.float64).transpose(0, 3, 1, 2)


def new_ws(dc, nbytes=None):
    return torch.zeros(max(nbytes or 0, dc.conv_workspace_bytes()), dtype=torch.uint8, device="cuda")


def run_merge(dc, specs, residuals, packed_dtype=None, algo=0):
    layers = [dc.DeviceLayer(s) for s in specs]
    g, ws_bytes = dc.merge_query(layers, residuals)
    bufs = [Guarded(torch, (g.c_out, g.c_in, g.k, g.k), torch.float32, fill=float("nan")),
            Guarded(torch, (g.c_out,), torch.float32, fill=float("nan")),
            Guarded(torch, (ws_bytes,), torch.uint8)]
    wm, bm, ws = (b.t for b in bufs)
    packed = None
    if packed_dtype is not None:
        bufs.append(Guarded(torch, (dc.packed_bytes(g, packed_dtype),), torch.uint8))
        packed = bufs[-1].t
    dc.merge_chain(layers, residuals, wm, bm, packed, packed_dtype if packed_dtype is not None else dc.F32, ws,
                   algo=algo)
    torch.cuda.synchronize()
    for b, name in zip(bufs, ("merged weights", "merged bias", "merge workspace", "packed weights")):
        b.check(name)
    assert not torch.isnan(wm).any() and not torch.isnan(bm).any()
    return g, wm, bm, packed


def run_conv(dc, x, g, packed, bias, act, residual=None, algo=0):
    n, h, w, _ = x.shape
    ho, wo = O.out_extent(h, g.k, g.stride, g.pad), O.out_extent(w, g.k, g.stride, g.pad)
    gy = Guarded(torch, (n, ho, wo, g.c_out), x.dtype, fill=float("nan"))
    gws = Guarded(torch, (dc.conv_workspace_bytes(),), torch.uint8, fill=0)
    y, ws = gy.t, gws.t
    dc.conv_forward(x, g, packed, bias, act, residual, y, ws, algo=algo)
    assert dc.workspace_status(ws) == dc.OK
    gy.check("conv output")
    gws.check("conv workspace")
    assert not torch.isnan(y.float()).any(), "an output element was never written"
    return y


def small_chain(name, rng_seed=0):
    """Reduced-size versions of the four single-span topologies plus harder ones."""
    mk = I.make_layer
    s = rng_seed
    if name == "t0":
        return [mk(s, 0, 16, 96, 1, 1, 0), mk(s, 1, 96, 96, 3, 1, 1, depthwise=True), mk(s, 2, 96, 24, 1, 1, 0)], []
    if name == "t1":
        return [mk(s, 0, 24, 144, 1, 1, 0), mk(s, 1, 144, 144, 3, 1, 1, depthwise=True), mk(s, 2, 144, 24, 1, 1, 0)], [(0, 2)]
    if name == "t2":
        return [mk(s, 0, 24, 144, 1, 1, 0), mk(s, 1, 144, 144, 3, 2, 1, depthwise=True), mk(s, 2, 144, 32, 1, 1, 0)], []
    if name == "t3":
        L = []
        for b in range(2):
            L += [mk(s, 3 * b, 32, 192, 1, 1, 0), mk(s, 3 * b + 1, 192, 192, 3, 1, 1, depthwise=True),
                  mk(s, 3 * b + 2, 192, 32, 1, 1, 0)]
        return L, [(0, 2), (3, 5)]
    if name == "dense_pair":
        return [mk(s, 0, 8, 16, 3, 1, 1), mk(s, 1, 16, 8, 3, 1, 1, with_bn=False)], []
    if name == "s2_first":
        return [mk(s, 0, 8, 16, 3, 2, 1), mk(s, 1, 16, 16, 1, 1, 0), mk(s, 2, 16, 24, 1, 1, 0)], []
    if name == "dw_first":
        return [mk(s, 0, 16, 16, 3, 1, 1, depthwise=True), mk(s, 1, 16, 16, 3, 1, 1, depthwise=True),
                mk(s, 2, 16, 8, 1, 1, 0)], [(0, 0)]
    if name == "dw_only":
        return [mk(s, 0, 8, 8, 3, 1, 1, depthwise=True), mk(s, 1, 8, 8, 3, 2, 1, depthwise=True)], []
    if name == "single":
        return [mk(s, 0, 8, 24, 3, 1, 1)], []
    if name == "skip_mid":
        return [mk(s, 0, 8, 16, 1, 1, 0), mk(s, 1, 16, 16, 3, 1, 1, depthwise=True), mk(s, 2, 16, 40, 1, 1, 0)], [(1, 1)]
    raise KeyError(name)


CHAINS = ["t0", "t1", "t2", "t3", "dense_pair", "s2_first", "dw_first", "dw_only", "single", "skip_mid"]


def test_fold_bn(dc):
    for spec in (I.make_layer(3, 0, 24, 40, 3, 1, 1), I.make_layer(3, 1, 32, 32, 3, 1, 1, depthwise=True),
                 I.make_layer(3, 2, 8, 8, 1, 1, 0, with_bn=False)):
        lay = dc.DeviceLayer(spec)
        w = torch.empty_like(lay.weight)
        b = torch.empty(spec.c_out, device="cuda")
        dc.fold_bn(lay, w, b)
        Wo, bo = O.fold_bn(spec)
        assert O.rel_l2(w.cpu().numpy(), Wo) < 1e-6 and O.rel_l2(b.cpu().numpy(), bo) < 1e-6 or \
            (spec.bn is None and np.all(bo == 0) and float(b.abs().max()) == 0)


@pytest.mark.parametrize("name", CHAINS)
def test_merge_chain_weights(dc, name):
    specs, res = small_chain(name)
    g, wm, bm, _ = run_merge(dc, specs, res)
    W, b, k, s, p = O.merge_formula(specs, res)
    assert (g.k, g.stride, g.pad, g.c_in, g.c_out) == (k, s, p, W.shape[1], W.shape[0])
    assert O.rel_l2(wm.cpu().numpy(), W) <= TOL_W
    assert O.rel_l2(bm.cpu().numpy(), b) <= TOL_W


def wide_chain(name, s=5):
    """Runs with more arithmetic than `small_chain`: two skip blocks in a row at three widths, a
    dense 3x3 o 3x3 o 3x3 run (7x7 result) and a stride-2 run with a 5x5 depthwise layer."""
    mk = I.make_layer
    if name in ("two_blocks_32", "two_blocks_64", "two_blocks_48"):
        c = int(name.rsplit("_", 1)[1])
        L = []
        for b in range(2):
            L += [mk(s, 3 * b, c, 6 * c, 1, 1, 0), mk(s, 3 * b + 1, 6 * c, 6 * c, 3, 1, 1, depthwise=True),
                  mk(s, 3 * b + 2, 6 * c, c, 1, 1, 0)]
        return L, [(0, 2), (3, 5)]
    if name == "dense_7x7":
        return [mk(s, 0, 16, 24, 3, 1, 1), mk(s, 1, 24, 24, 3, 1, 1), mk(s, 2, 24, 16, 3, 1, 1)], [(1, 1)]
    if name == "s2_dw5":
        return [mk(s, 0, 40, 240, 1, 1, 0), mk(s, 1, 240, 240, 5, 2, 2, depthwise=True), mk(s, 2, 240, 48, 1, 1, 0)], []
    raise KeyError(name)


WIDE = ["two_blocks_32", "two_blocks_64", "two_blocks_48", "dense_7x7", "s2_dw5"]


@pytest.mark.parametrize("algo", ["steps", "auto"])
@pytest.mark.parametrize("name", CHAINS + WIDE)
def test_merge_chain_both_walks(dc, name, algo):
    """The pairwise walk and the walk that merges inverted-residual blocks in one step, each
    against the oracle's formula (weights, bias, and the bf16 packed copy through the fp32 result)."""
    specs, res = small_chain(name) if name in CHAINS else wide_chain(name)
    code = dc.MERGE_STEPS if algo == "steps" else dc.MERGE_AUTO
    g, wm, bm, packed = run_merge(dc, specs, res, packed_dtype=dc.BF16, algo=code)
    W, b, k, s, p = O.merge_formula(specs, res)
    assert (g.k, g.stride, g.pad) == (k, s, p)
    assert O.rel_l2(wm.cpu().numpy(), W) <= TOL_W
    assert O.rel_l2(bm.cpu().numpy(), b) <= TOL_W
    # the packed copy must be what dc_pack_weights makes of the delivered fp32 kernel, bit for bit
    again = torch.empty_like(packed)
    dc.pack_weights(wm, g, dc.BF16, again)
    torch.cuda.synchronize()
    assert torch.equal(packed, again)


@pytest.mark.parametrize("case", ["no_bn", "bias_no_bn", "wide_hidden", "block_inside_run", "fold_order", "rows_order",
                                  "block_after_1x1", "skip_1x1_then_3x3"])
def test_block_step_edge_cases(dc, case):
    """Blocks without BN, with plain biases, with a hidden width that is staged in several passes,
    and a block in the middle of a longer run (neighbours composed pairwise around it)."""
    mk = I.make_layer
    if case == "no_bn":
        specs = [mk(11, 0, 8, 48, 1, 1, 0, with_bn=False), mk(11, 1, 48, 48, 3, 1, 1, depthwise=True, with_bn=False),
                 mk(11, 2, 48, 8, 1, 1, 0, with_bn=False)]
        res = [(0, 2)]
    elif case == "bias_no_bn":
        specs = [mk(12, 0, 16, 96, 1, 1, 0, with_bn=False, with_bias=True),
                 mk(12, 1, 96, 96, 5, 2, 2, depthwise=True), mk(12, 2, 96, 24, 1, 1, 0, with_bias=True)]
        res = []
    elif case == "wide_hidden":
        specs = [mk(13, 0, 160, 960, 1, 1, 0), mk(13, 1, 960, 960, 3, 1, 1, depthwise=True), mk(13, 2, 960, 160, 1, 1, 0)]
        res = [(0, 2)]
    elif case == "block_after_1x1":  # a k x k piece composed after a 1x1 layer: one term per tap sum
        specs = [mk(17, 0, 40, 16, 1, 1, 0), mk(17, 1, 16, 96, 1, 1, 0), mk(17, 2, 96, 96, 3, 1, 1, depthwise=True),
                 mk(17, 3, 96, 16, 1, 1, 0)]
        res = [(1, 3)]
    elif case == "skip_1x1_then_3x3":  # (W1 + I) under a dense 3x3
        specs = [mk(18, 0, 24, 24, 1, 1, 0), mk(18, 1, 24, 40, 3, 1, 1)]
        res = [(0, 0)]
    elif case == "fold_order":      # 40-64 input channels, narrow output: packed copy in the fold order
        specs = [mk(15, 0, 48, 288, 1, 1, 0), mk(15, 1, 288, 288, 3, 1, 1, depthwise=True), mk(15, 2, 288, 24, 1, 1, 0)]
        res = []
    elif case == "rows_order":      # wide input and output: packed copy in 64-channel planes
        specs = [mk(16, 0, 64, 384, 1, 1, 0), mk(16, 1, 384, 384, 3, 1, 1, depthwise=True), mk(16, 2, 384, 64, 1, 1, 0)]
        res = [(0, 2)]
    else:
        specs = [mk(14, 0, 16, 8, 3, 1, 1), mk(14, 1, 8, 48, 1, 1, 0), mk(14, 2, 48, 48, 3, 1, 1, depthwise=True),
                 mk(14, 3, 48, 8, 1, 1, 0), mk(14, 4, 8, 24, 1, 1, 0)]
        res = [(1, 3)]
    g, wm, bm, packed = run_merge(dc, specs, res, packed_dtype=dc.BF16)
    W, b, *_ = O.merge_formula(specs, res)
    assert O.rel_l2(wm.cpu().numpy(), W) <= TOL_W
    assert O.rel_l2(bm.cpu().numpy(), b) <= TOL_W
    again = torch.empty_like(packed)
    dc.pack_weights(wm, g, dc.BF16, again)
    torch.cuda.synchronize()
    assert torch.equal(packed, again)
    g2, wm2, bm2, _ = run_merge(dc, specs, res, algo=dc.MERGE_STEPS)
    assert O.rel_l2(wm2.cpu().numpy(), W) <= TOL_W and O.rel_l2(bm2.cpu().numpy(), b) <= TOL_W


@pytest.mark.parametrize("case", ["expand_dw", "dw_project", "dw_s2_project", "dw_skip_project", "expand_skip_dw", "whole_skip",
                                  "no_bn", "narrow", "dense_pair_skips", "dense_pair_ragged", "block_ragged", "block_k5",
                                  "wide_1x1_pair"])
def test_runs_delivered_by_one_launch(dc, case):
    """Runs whose merge and delivery are one launch (a block, two dense 3x3 layers, a 1x1 and a depthwise layer), at ragged
    tile edges, with identities on one layer or on the whole run, and the fp32 packed copy as well."""
    mk = I.make_layer
    res = []
    if case == "expand_dw":
        specs = [mk(51, 0, 24, 104, 1, 1, 0), mk(51, 1, 104, 104, 3, 2, 1, depthwise=True)]
    elif case == "dw_project":
        specs = [mk(52, 0, 136, 136, 3, 1, 1, depthwise=True), mk(52, 1, 136, 40, 1, 1, 0)]
    elif case == "dw_s2_project":
        specs = [mk(53, 0, 56, 56, 3, 2, 1, depthwise=True), mk(53, 1, 56, 264, 1, 1, 0)]
    elif case == "dw_skip_project":
        specs, res = [mk(54, 0, 48, 48, 3, 1, 1, depthwise=True), mk(54, 1, 48, 24, 1, 1, 0)], [(0, 0)]
    elif case == "expand_skip_dw":
        specs, res = [mk(55, 0, 40, 40, 1, 1, 0), mk(55, 1, 40, 40, 3, 1, 1, depthwise=True)], [(0, 0), (1, 1)]
    elif case == "whole_skip":
        specs, res = [mk(56, 0, 72, 72, 3, 1, 1, depthwise=True), mk(56, 1, 72, 72, 1, 1, 0)], [(0, 1)]
    elif case == "no_bn":
        specs = [mk(57, 0, 16, 32, 1, 1, 0, with_bn=False, with_bias=True), mk(57, 1, 32, 32, 3, 1, 1, depthwise=True, with_bn=False)]
    elif case == "narrow":           # channels that are no multiple of a packed chunk
        specs = [mk(58, 0, 6, 20, 1, 1, 0), mk(58, 1, 20, 20, 3, 1, 1, depthwise=True)]
    elif case == "dense_pair_skips":
        specs, res = [mk(59, 0, 24, 24, 3, 1, 1), mk(59, 1, 24, 24, 3, 1, 1)], [(0, 0), (1, 1)]
    elif case == "dense_pair_ragged":
        specs, res = [mk(60, 0, 20, 44, 3, 1, 1), mk(60, 1, 44, 13, 3, 2, 1, with_bn=False)], []
    elif case == "block_ragged":
        specs = [mk(61, 0, 40, 92, 1, 1, 0), mk(61, 1, 92, 92, 3, 2, 1, depthwise=True), mk(61, 2, 92, 21, 1, 1, 0)]
    elif case == "block_k5":
        specs = [mk(62, 0, 24, 64, 1, 1, 0), mk(62, 1, 64, 64, 5, 1, 2, depthwise=True), mk(62, 2, 64, 24, 1, 1, 0)]
        res = [(0, 2)]
    else:
        specs = [mk(63, 0, 320, 96, 1, 1, 0), mk(63, 1, 96, 640, 1, 1, 0)]
    W, b, k, s, p = O.merge_formula(specs, res)
    for code in (dc.BF16, dc.F32):
        g, wm, bm, packed = run_merge(dc, specs, res, packed_dtype=code)
        assert (g.k, g.stride, g.pad) == (k, s, p)
        assert O.rel_l2(wm.cpu().numpy(), W) <= TOL_W and O.rel_l2(bm.cpu().numpy(), b) <= TOL_W
        again = torch.full_like(packed, 7)
        dc.pack_weights(wm, g, code, again)
        torch.cuda.synchronize()
        assert torch.equal(packed, again)


@pytest.mark.parametrize("channels,res,bn", [
    ((8, 4, 8), [], True),                     # one piece of four channels: three of four groups have no slice
    ((36, 20, 44), [], True),                  # nothing a multiple of a tile or of a slice
    ((40, 40, 40), [(0, 0)], True),            # an identity on the first layer, ...
    ((40, 40, 40), [(0, 0), (1, 1)], False),   # ... on both, ...
    ((72, 24, 72), [(0, 1)], True),            # ... on the run
    ((648, 72, 712), [], True),                # tiles of 64 columns, ragged ones last
    ((960, 320, 1280), [], True),              # the network's last merge: tiles of 48 rows
])
def test_two_1x1_layers_delivered_by_one_launch(dc, channels, res, bn):
    a, m, o = channels
    specs = [I.make_layer(81, 0, a, m, 1, 1, 0, with_bn=bn), I.make_layer(81, 1, m, o, 1, 1, 0)]
    _check_delivery(dc, specs, res, (dc.BF16, dc.F32) if a % 8 == 0 and o % 8 == 0 else (dc.F32,))


@pytest.mark.parametrize("c0,c1,c2,s,res", [
    (40, 36, 24, 1, []),                       # a slice of 4 channels last, ragged tiles
    (32, 32, 32, 1, [(0, 0)]),                 # an identity on the 1x1 layer, ...
    (32, 32, 32, 1, [(0, 0), (1, 1)]),         # ... and on the 3x3 one
    (384, 96, 100, 2, []),                     # three slices, stride 2
    (72, 200, 9, 1, []),                       # one output channel more than a tile
])
@pytest.mark.parametrize("tail", [False, True])
def test_3x3_after_1x1_against_the_oracle(dc, c0, c1, c2, s, res, tail):
    """As a run's last composition, delivered by its own launch, and as a piece that a depthwise layer is composed with."""
    specs = [I.make_layer(82, 0, c0, c1, 1, 1, 0), I.make_layer(82, 1, c1, c2, 3, s, 1)]
    if tail:
        specs.append(I.make_layer(82, 2, c2, c2, 3, 1, 1, depthwise=True))
    _check_delivery(dc, specs, res, (dc.BF16, dc.F32))


def test_3x3_after_1x1_with_more_outputs_than_a_grid_has_rows(dc):
    """65544 output channels: a grid with a row for each, as the kernel for fewer intermediate channels has, is refused."""
    _check_delivery(dc, [I.make_layer(85, 0, 8, 32, 1, 1, 0), I.make_layer(85, 1, 32, 65544, 3, 1, 1)], [], (dc.BF16, dc.F32))


def _check_delivery(dc, specs, res, codes):
    W, b, k, s, p = O.merge_formula(specs, res)
    for code in codes:
        g, wm, bm, packed = run_merge(dc, specs, res, packed_dtype=code)
        assert (g.k, g.stride, g.pad) == (k, s, p)
        assert O.rel_l2(wm.cpu().numpy(), W) <= TOL_W and O.rel_l2(bm.cpu().numpy(), b) <= TOL_W
        again = torch.full_like(packed, 7)
        dc.pack_weights(wm, g, code, again)
        torch.cuda.synchronize()
        assert torch.equal(packed, again)


@pytest.mark.parametrize("c,hidden", [(24, 320), (136, 820), (160, 960), (200, 1000)])
def test_blocks_by_sixteen_warps_against_the_oracle(dc, c, hidden):
    """Long reductions: tiles of 8 x 16 and of 8 x 24 pairs, warps whose last slice is short or that have none."""
    _check_delivery(dc, [I.make_layer(83, 0, c, hidden, 1, 1, 0), I.make_layer(83, 1, hidden, hidden, 3, 1, 1, depthwise=True),
                         I.make_layer(83, 2, hidden, c, 1, 1, 0)], [(0, 2)], (dc.BF16, dc.F32))


@pytest.mark.parametrize("a,c,o,res", [(152, 4, 160, []), (160, 20, 148, []), (148, 36, 152, []), (152, 152, 152, [(0, 0), (1, 1)]),
                                       (152, 152, 152, [(0, 1)]), (200, 132, 256, [])])
def test_3x3_after_3x3_by_four_warps_against_the_oracle(dc, a, c, o, res):
    """More tiles than two to an SM: warps with two parts of the reduction, with one, with one that is cut short, with none."""
    _check_delivery(dc, [I.make_layer(84, 0, a, c, 3, 1, 1), I.make_layer(84, 1, c, o, 3, 1, 1)], res,
                    (dc.BF16, dc.F32) if a % 8 == 0 and o % 8 == 0 else (dc.F32,))


@pytest.mark.parametrize("case", ["block", "dense_pair", "expand_dw"])
@pytest.mark.parametrize("alias", ["weights", "bias", "packed"])
def test_merge_into_its_layers_arrays(dc, case, alias):
    """Outputs that lie where the layers' arrays lie: the same result as into buffers of their own."""
    mk = I.make_layer
    specs = {"block": [mk(71, 0, 40, 240, 1, 1, 0), mk(71, 1, 240, 240, 3, 1, 1, depthwise=True), mk(71, 2, 240, 40, 1, 1, 0)],
             "dense_pair": [mk(72, 0, 64, 64, 3, 1, 1), mk(72, 1, 64, 64, 3, 1, 1)],
             "expand_dw": [mk(73, 0, 96, 96, 1, 1, 0), mk(73, 1, 96, 96, 3, 1, 1, depthwise=True)]}[case]
    g, wm, bm, packed = run_merge(dc, specs, [], packed_dtype=dc.BF16)
    layers = [dc.DeviceLayer(s) for s in specs]
    _, ws_bytes = dc.merge_query(layers, [])
    ws = torch.zeros(ws_bytes, dtype=torch.uint8, device="cuda")
    out = {"weights": torch.empty_like(wm), "bias": torch.empty_like(bm), "packed": torch.empty_like(packed)}
    # the layer's array lies at the start of the output's buffer
    last = layers[-1] if alias == "bias" and case == "block" else layers[0]
    src = last.bn[1] if alias == "bias" else last.weight
    flat = out[alias].reshape(-1).view(torch.uint8).view(torch.float32)
    assert flat.numel() >= src.numel()
    flat[:src.numel()].copy_(src.reshape(-1))
    if alias == "bias":
        last.c.bn_beta = flat.data_ptr()
    else:
        last.c.weight = flat.data_ptr()
    dc.merge_chain(layers, [], out["weights"], out["bias"], out["packed"], dc.BF16, ws)
    torch.cuda.synchronize()
    # two walks of the same fp32 sums: a few units of the last place apart
    assert O.rel_l2(out["weights"].cpu().numpy(), wm.cpu().numpy()) <= 1e-6 and O.rel_l2(out["bias"].cpu().numpy(), bm.cpu().numpy()) <= 1e-6
    again = torch.empty_like(packed)
    dc.pack_weights(out["weights"], g, dc.BF16, again)
    assert torch.equal(out["packed"], again)


@pytest.mark.parametrize("specs,bound", [
    ([(160, 960, 1, 0), (960, 960, 3, 1), (960, 160, 1, 0)], 2.7e-7),
    ([(64, 64, 3, 1), (64, 64, 3, 1)], 2.1e-7),
])
def test_merges_sum_in_parts(dc, specs, bound):
    """The one-launch merges add up eight partial sums: their error against 64 bits (1.8e-7 and 1.4e-7 measured) stays clear
    of what one running sum over all intermediate channels shows (4.5e-7 and 3.1e-7); the bound lies half way down."""
    layers = [I.make_layer(74, i, ci, co, k, 1, p, depthwise=ci == co == 960) for i, (ci, co, k, p) in enumerate(specs)]
    g, wm, bm, _ = run_merge(dc, layers, [])
    W, b, *_ = O.merge_formula(layers, [])
    assert O.rel_l2(wm.cpu().numpy(), W) <= bound and O.rel_l2(bm.cpu().numpy(), b) <= 3e-7


def test_a_launch_that_is_refused_is_reported(dc):
    """A 3x3 layer with 65536 outputs after a 1x1 layer needs a grid the device does not have (the runtime refuses the
    launch, nothing runs).  The 1x1 layer after it is composed by the fp32 convolution, whose launch succeeds: the merge
    must report the refused one all the same.  Asked once more, the library has no error left over."""
    z = lambda *s: torch.zeros(*s, device="cuda")
    shapes = [(64, 4, 1, 0), (4, 65536, 3, 1), (65536, 352, 1, 0)]
    keep = [z(co, ci, k, k) for ci, co, k, _ in shapes]
    layers = [dc.Layer(ci, co, 1, k, 1, p, w.data_ptr(), None, None, None, None, None, 0.0) for (ci, co, k, p), w in zip(shapes, keep)]
    g, ws_bytes = dc.merge_query(layers, [])
    wm, bm, ws = z(g.c_out, g.c_in, 3, 3), z(g.c_out), torch.zeros(ws_bytes, dtype=torch.uint8, device="cuda")
    with pytest.raises(dc.DcError) as e:
        dc.merge_chain(layers, [], wm, bm, None, dc.F32, ws)
    assert e.value.status == dc.ERR_CUDA
    torch.cuda.synchronize()
    del keep, layers, wm, bm, ws
    specs, res = small_chain("t1")
    g, wm, bm, _ = run_merge(dc, specs, res)
    assert O.rel_l2(wm.cpu().numpy(), O.merge_formula(specs, res)[0]) <= TOL_W


@pytest.mark.parametrize("c,n,h,w", [(64, 2, 28, 28), (128, 2, 14, 14), (256, 1, 14, 14), (512, 1, 14, 14)])
def test_vgg_style_dense_merge(dc, c, n, h, w):
    """Two dense 3x3 layers (VGG-style, c -> c -> c) merged into one 5x5 layer: merged weights against
    the formula, and the bf16 forward of the merged layer (tensor-bound for these widths) against the
    sequential chain."""
    mk = I.make_layer
    specs = [mk(31, 0, c, c, 3, 1, 1), mk(31, 1, c, c, 3, 1, 1)]
    g, wm, bm, packed = run_merge(dc, specs, [], packed_dtype=dc.BF16)
    assert (g.k, g.stride, g.pad) == (5, 1, 2)
    W, b, *_ = O.merge_formula(specs, [])
    assert O.rel_l2(wm.cpu().numpy(), W) <= TOL_W and O.rel_l2(bm.cpu().numpy(), b) <= TOL_W
    assert dc.conv_kernel_name(n, h, w, g, dc.BF16) == "k_conv_tc_rows"
    x = I.make_input(32, (n, h, w, c), bf16=True)
    y = run_conv(dc, dev(x, torch.bfloat16), g, packed, bm, dc.ACT_IDENTITY)
    ref = O.chain_forward_reordered(x.transpose(0, 3, 1, 2), specs, [])
    assert_close(nchw(y), ref, TOL_BF16)


def width14_chain(name, s=41):
    """Spans with the channel counts of MobileNetV2 at width 1.4 (Fig. 4: 48, 24, 32, 144, ...)."""
    mk = I.make_layer
    if name == "first_block":      # depthwise 48 + projection to 24 (t = 1 block after the 48-channel stem)
        return [mk(s, 0, 48, 48, 3, 1, 1, depthwise=True), mk(s, 1, 48, 24, 1, 1, 0)], []
    if name == "block_s2":         # 24 -> 144 -> 32, stride 2
        return [mk(s, 0, 24, 144, 1, 1, 0), mk(s, 1, 144, 144, 3, 2, 1, depthwise=True), mk(s, 2, 144, 32, 1, 1, 0)], []
    if name == "block_res_32":     # 32 -> 192 -> 32 with its skip folded
        return [mk(s, 0, 32, 192, 1, 1, 0), mk(s, 1, 192, 192, 3, 1, 1, depthwise=True), mk(s, 2, 192, 32, 1, 1, 0)], [(0, 2)]
    if name == "block_res_88":     # 88 -> 528 -> 88 (64 x 1.4 rounded to 8)
        return [mk(s, 0, 88, 528, 1, 1, 0), mk(s, 1, 528, 528, 3, 1, 1, depthwise=True), mk(s, 2, 528, 88, 1, 1, 0)], [(0, 2)]
    if name == "cross_block_48":   # two 48-channel blocks merged across their boundary: 5x5, 48 -> 48
        L = []
        for b in range(2):
            L += [mk(s, 3 * b, 48, 288, 1, 1, 0), mk(s, 3 * b + 1, 288, 288, 3, 1, 1, depthwise=True),
                  mk(s, 3 * b + 2, 288, 48, 1, 1, 0)]
        return L, [(0, 2), (3, 5)]
    if name == "project_expand":   # projection of one block and expansion of the next: 144 -> 32 -> 192
        return [mk(s, 0, 144, 32, 1, 1, 0), mk(s, 1, 32, 192, 1, 1, 0)], []
    raise KeyError(name)


@pytest.mark.parametrize("name,n,h,w", [("first_block", 2, 28, 28), ("block_s2", 2, 28, 28), ("block_res_32", 2, 28, 28),
                                        ("block_res_88", 2, 14, 14), ("cross_block_48", 2, 14, 14),
                                        ("project_expand", 1, 14, 14)])
def test_width_1p4_spans(dc, name, n, h, w):
    """Merge and bf16 forward of spans at MobileNetV2-1.4 widths, both walks of the merge."""
    specs, res = width14_chain(name)
    W, b, k, s, p = O.merge_formula(specs, res)
    for algo in (dc.MERGE_AUTO, dc.MERGE_STEPS):
        g, wm, bm, packed = run_merge(dc, specs, res, packed_dtype=dc.BF16, algo=algo)
        assert (g.k, g.stride, g.pad) == (k, s, p)
        assert O.rel_l2(wm.cpu().numpy(), W) <= TOL_W and O.rel_l2(bm.cpu().numpy(), b) <= TOL_W
    x = I.make_input(42, (n, h, w, specs[0].c_in), bf16=True)
    y = run_conv(dc, dev(x, torch.bfloat16), g, packed, bm, dc.ACT_RELU6)
    ref = O.chain_forward_reordered(x.transpose(0, 3, 1, 2), specs, res, final_act="relu6")
    assert_close(nchw(y), ref, TOL_BF16, what=name)


@pytest.mark.parametrize("stride", [1, 2])
def test_large_packed_copy_is_written_chunk_by_chunk(dc, stride):
    """Merged kernels whose packed copy has 262 144 elements or more are packed one 16-byte chunk per
    thread (rows order for stride 1, general order for stride 2): same bits as dc_pack_weights."""
    mk = I.make_layer
    specs = [mk(21, 0, 192, 192, 1, 1, 0), mk(21, 1, 192, 192, 3, stride, 1)]
    g, wm, bm, packed = run_merge(dc, specs, [], packed_dtype=dc.BF16)
    assert packed.numel() // 2 >= 262144
    W, b, *_ = O.merge_formula(specs, [])
    assert O.rel_l2(wm.cpu().numpy(), W) <= TOL_W and O.rel_l2(bm.cpu().numpy(), b) <= TOL_W
    again = torch.empty_like(packed)
    dc.pack_weights(wm, g, dc.BF16, again)
    torch.cuda.synchronize()
    assert torch.equal(packed, again)


@pytest.mark.parametrize("name", CHAINS)
def test_merged_conv_fp32_equals_sequential_chain(dc, name):
    specs, res = small_chain(name, rng_seed=1)
    g, wm, bm, packed = run_merge(dc, specs, res, packed_dtype=dc.F32)
    x = I.make_input(1, (2, 13, 11, specs[0].c_in))
    y = run_conv(dc, dev(x), g, packed, bm, dc.ACT_IDENTITY)
    ref = O.chain_forward_reordered(x.transpose(0, 3, 1, 2), specs, res)
    assert y.shape[1:3] == ref.shape[2:]
    assert_close(nchw(y), ref, TOL_F32, bf16=False)


def test_config0_tiny_fp32(dc):
    case = I.chain_case(0)
    g, wm, bm, packed = run_merge(dc, case.layers, case.residuals, packed_dtype=dc.F32)
    W, b, k, s, p = O.merge_formula(case.layers, case.residuals)
    assert (g.c_in, g.c_out, g.k, g.stride, g.pad) == (16, 24, 3, 1, 1)
    assert O.rel_l2(wm.cpu().numpy(), W) <= TOL_W and O.rel_l2(bm.cpu().numpy(), b) <= TOL_W
    x = case.x()
    y = run_conv(dc, dev(x), g, packed, bm, dc.ACT_IDENTITY)
    ref = O.chain_forward_reordered(x.transpose(0, 3, 1, 2), case.layers, case.residuals)
    assert_close(nchw(y), ref, TOL_F32, bf16=False)
    # the chain with its original per-layer padding agrees inside and differs on the border ring
    orig = O.chain_forward_original(x.transpose(0, 3, 1, 2), case.layers, case.residuals)
    assert O.rel_l2(nchw(y)[:, :, 1:-1, 1:-1], orig[:, :, 1:-1, 1:-1]) <= TOL_F32
    assert O.rel_l2(nchw(y), orig) > 1e-3


BF16_SHAPES = [
    # (name, n, h, w) -- spatial sizes that span several tiles and leave ragged tails
    ("t1", 3, 19, 23), ("t2", 2, 22, 18), ("t3", 2, 17, 21), ("t0", 1, 9, 40), ("s2_first", 2, 30, 14),
    ("dense_pair", 2, 12, 70), ("single", 3, 8, 8), ("skip_mid", 1, 33, 9),
]


@pytest.mark.parametrize("algo", ["simt", "auto"])
@pytest.mark.parametrize("name,n,h,w", BF16_SHAPES)
def test_merged_conv_bf16_equals_sequential_chain(dc, name, n, h, w, algo):
    specs, res = small_chain(name, rng_seed=2)
    g, wm, bm, packed = run_merge(dc, specs, res, packed_dtype=dc.BF16)
    x = I.make_input(2, (n, h, w, specs[0].c_in), bf16=True)
    for act in (dc.ACT_IDENTITY, dc.ACT_RELU6):
        y = run_conv(dc, dev(x, torch.bfloat16), g, packed, bm, act,
                     algo=dc.ALGO_SIMT if algo == "simt" else dc.ALGO_AUTO)
        ref = O.chain_forward_reordered(x.transpose(0, 3, 1, 2), specs, res,
                                        final_act="relu6" if act else None)
        assert not torch.isnan(y.float()).any()
        assert_close(nchw(y), ref, TOL_BF16)


@pytest.mark.parametrize("algo", ["simt", "auto"])
@pytest.mark.parametrize("c_in,c_out,k,s,p,n,h,w", [
    (32, 16, 1, 1, 0, 2, 14, 14), (96, 24, 1, 1, 0, 1, 20, 12), (160, 320, 1, 1, 0, 2, 7, 7),
    (320, 1280, 1, 1, 0, 1, 7, 7), (3, 32, 3, 2, 1, 2, 32, 32), (16, 96, 1, 1, 0, 1, 24, 24),
    (96, 144, 5, 2, 2, 1, 20, 20), (64, 384, 1, 1, 0, 3, 14, 14), (24, 40, 7, 1, 3, 1, 16, 16),
    (40, 24, 3, 1, 0, 1, 12, 12), (20, 12, 3, 1, 1, 1, 10, 10),
])
def test_single_conv_bf16_with_explicit_skip(dc, c_in, c_out, k, s, p, n, h, w, algo):
    spec = I.make_layer(5, 0, c_in, c_out, k, s, p)
    lay = dc.DeviceLayer(spec)
    wf = torch.empty_like(lay.weight)
    bf = torch.empty(c_out, device="cuda")
    dc.fold_bn(lay, wf, bf)
    g = dc.geom(c_in, c_out, 1, k, s, p)
    packed = torch.empty(dc.packed_bytes(g, dc.BF16), dtype=torch.uint8, device="cuda")
    dc.pack_weights(wf, g, dc.BF16, packed)
    x = I.make_input(6, (n, h, w, c_in), bf16=True)
    ho, wo = O.out_extent(h, k, s, p), O.out_extent(w, k, s, p)
    r = I.round_bf16(I.normal(7, 99, (n, ho, wo, c_out)))
    y = run_conv(dc, dev(x, torch.bfloat16), g, packed, bf, dc.ACT_RELU6, residual=dev(r, torch.bfloat16),
                 algo=dc.ALGO_SIMT if algo == "simt" else dc.ALGO_AUTO)
    Wf, bfo = O.fold_bn(spec)
    ref = O.relu6(O.conv_direct(x.transpose(0, 3, 1, 2), Wf, bfo, k, s, p) + r.transpose(0, 3, 1, 2))
    assert_close(nchw(y), ref, TOL_BF16)


# One case per branch of the forward kernels: the expected kernel is asserted, so a change of the
# dispatch rules cannot silently drop a kernel from the parity suite.
@pytest.mark.parametrize("c_in,c_out,k,s,p,n,h,w,kernel", [
    (24, 24, 3, 1, 1, 3, 30, 22, "k_conv_tc_pairrows"),     # odd padding: pairs (2j-1, 2j), masked ends
    (32, 32, 5, 1, 2, 2, 28, 28, "k_conv_tc_pairrows"),     # 5x5, even padding, full 128-byte lines
    (16, 8, 3, 1, 0, 1, 18, 40, "k_conv_tc_pairrows"),      # no padding, 16 of 64 channels of a line used
    (8, 16, 3, 1, 1, 1, 6, 300, "k_conv_tc_pairrows"),      # three column strips: per-pixel stores, strip halos
    (16, 16, 7, 1, 3, 1, 20, 20, "k_conv_tc_pairrows"),     # 7x7: 56 instructions per block
    (24, 24, 3, 1, 1, 1, 9, 15, "k_conv_tc_pairrows"),      # odd width, one small image
    (40, 32, 5, 1, 2, 2, 14, 14, "k_conv_tc_fold"),         # odd entry count (padding entry), 5 tap columns
    (48, 24, 3, 1, 1, 2, 20, 20, "k_conv_tc_fold"),
    (64, 32, 3, 1, 1, 1, 12, 70, "k_conv_tc_fold"),         # two column strips
    (4, 16, 5, 1, 2, 1, 9, 200, "k_conv_stem_tc"),          # two row segments per output row, 26 chunk planes
    (3, 40, 3, 2, 1, 2, 17, 33, "k_conv_stem_tc"),          # 40 output channels (48 operand rows), odd sizes
    (3, 32, 3, 2, 1, 3, 40, 300, "k_conv_stem_tc"),         # the stem's geometry, ragged second segment
    (1, 8, 3, 1, 1, 2, 20, 20, "k_conv_stem_tc"),           # one input channel
    (3, 24, 5, 2, 2, 2, 21, 304, "k_conv_stem_tc"),         # 16-byte row chunks with a shifted second segment
    (3, 32, 3, 2, 1, 2, 224, 224, "k_conv_stem_s2"),        # the stem itself: image rows as the operand, bands of 4 rows
    (3, 32, 3, 2, 1, 3, 41, 304, "k_conv_stem_s2"),         # two segments per output row (the second ragged), odd height
    (3, 40, 3, 2, 1, 2, 17, 32, "k_conv_stem_s2"),          # 40 output channels (48 operand rows), last band partial
    (4, 16, 3, 2, 0, 2, 20, 40, "k_conv_stem_s2"),          # no padding, four channels: pixels already 8 bytes
    (1, 8, 3, 2, 1, 2, 21, 24, "k_conv_stem_s2"),           # one input channel
    (2, 128, 3, 2, 1, 1, 12, 16, "k_conv_stem_s2"),         # 128 output channels: one output row per band
    (3, 32, 3, 2, 1, 64, 66, 64, "k_conv_stem_s2"),         # more bands than resident CTAs: one or two bands per CTA
    (3, 264, 3, 2, 1, 1, 20, 20, "k_conv_smallcin_bf16"),   # too many outputs for one accumulator: CUDA cores
    (24, 32, 3, 2, 1, 2, 28, 28, "k_conv_tc_pairrows"),     # stride 2: one output per line, even/odd row boxes
    (32, 16, 5, 2, 2, 1, 30, 44, "k_conv_tc_pairrows"),     # stride 2, even padding, 5x5
    (16, 24, 3, 2, 0, 2, 17, 36, "k_conv_tc_pairrows"),     # stride 2, no padding, odd height
    (40, 32, 3, 2, 1, 2, 28, 28, "k_conv_tc_rows_s2"),       # stride 2 by sub-tiles (more than 32 channels)
    (96, 144, 5, 2, 2, 1, 56, 56, "k_conv_tc_rows_s2"),      # the widest stride-2 merged layer of the network: several tiles per image
    (48, 64, 7, 2, 3, 1, 31, 44, "k_conv_tc_rows_s2"),       # 7x7 stride 2, odd height
    (48, 24, 5, 2, 1, 2, 22, 26, "k_conv_tc_rows_s2"),       # 5x5 stride 2 with padding 1
    (72, 48, 3, 2, 0, 1, 17, 150, "k_conv_tc_rows_s2"),      # stride 2 without padding, four column strips
    (32, 16, 1, 1, 0, 2, 20, 24, "k_conv_tc_pairrows"),     # 1x1: one instruction per 32-byte K step
    (32, 96, 1, 1, 0, 2, 20, 24, "k_conv_tc_rows"),         # 1x1 expansion from few channels: one half-filled plane
    (16, 96, 1, 1, 0, 1, 40, 112, "k_conv_tc_rows"),        # 1x1 expansion from 16 channels: one run of pixels, runs cut by blocks
    (32, 192, 3, 1, 1, 2, 28, 28, "k_conv_tc_rows"),        # 3x3 from few channels to more outputs than the pair rows take: two column strips, two passes
    (16, 136, 5, 1, 2, 1, 12, 20, "k_conv_tc_rows"),        # the same with 16 channels and a 5x5 kernel, two passes
    (32, 40, 1, 1, 0, 2, 20, 24, "k_conv_tc"),              # 1x1 with 40 outputs: general kernel
    (16, 128, 3, 1, 1, 1, 12, 16, "k_conv_tc_pairrows"),    # N = 256: two accumulator slots, run-time channel loop
    (32, 64, 3, 2, 1, 1, 28, 28, "k_conv_tc_pairrows"),     # stride 2, 64 output channels
    (160, 200, 3, 1, 1, 5, 7, 7, "k_conv_tc_rows"),         # three planes (the last half full), two passes; few images: one per tile, two strips, the reduction shared by three CTAs
    (96, 64, 1, 1, 0, 7, 7, 7, "k_conv_tc_rows"),           # 1x1 at 7 x 7, few images: a run of 343 pixels in three tiles
    (96, 64, 1, 1, 0, 733, 7, 7, "k_conv_tc_rows"),         # 1x1, a run of 35917 pixels: 141 tiles of 256, whatever image they lie in
    (160, 200, 3, 1, 1, 300, 7, 7, "k_conv_tc_rows"),       # 3x3 at 7 x 7 with more items than CTAs: three images per tile, two passes, runs cut by blocks (items shared by two CTAs)
    (960, 160, 1, 1, 0, 128, 7, 7, "k_conv_tc_rows"),       # deep projection of the network: tiles of 128 pixels, two passes of 80 channels
    (512, 512, 1, 1, 0, 6, 7, 7, "k_conv_tc_rows"),          # deep 1x1 with more than 256 outputs: two passes of 256 channels, one accumulator set
    (64, 48, 5, 1, 2, 1, 20, 70, "k_conv_tc_rows"),         # 5x5, tiles of one output row, the reduction shared by three CTAs
    (384, 64, 3, 1, 1, 2, 14, 14, "k_conv_tc_rows"),        # six planes, the reduction shared by five CTAs
    (128, 128, 5, 1, 2, 2, 14, 14, "k_conv_tc_rows"),       # 5x5 with 128 outputs in one pass, the reduction shared by six CTAs
    (96, 96, 7, 1, 3, 1, 14, 14, "k_conv_tc_rows"),         # 7x7: weight stages of one tap column, the reduction shared by eight CTAs
    (144, 32, 3, 1, 1, 1, 28, 28, "k_conv_tc_rows"),        # many channels, 32 outputs: the reduction shared by three CTAs
    (80, 48, 3, 1, 1, 2, 14, 27, "k_conv_tc_rows"),         # three strips of nine columns, resident weights
    (64, 64, 3, 1, 1, 1, 33, 45, "k_conv_tc_rows"),         # five strips of nine columns, row tiles of 11, resident weights
    (200, 24, 3, 1, 1, 2, 14, 14, "k_conv_tc"),             # many channels, fewer than 32 outputs: general kernel
    (192, 32, 1, 1, 0, 2, 28, 28, "k_conv_tc_rows"),        # 1x1 projection to 32 channels
])
def test_each_forward_kernel_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w, kernel, algo=0):
    g = dc.geom(c_in, c_out, 1, k, s, p)
    assert kernel is None or dc.conv_kernel_name(n, h, w, g, dc.BF16) == kernel
    spec = I.make_layer(11, 0, c_in, c_out, k, s, p)
    lay = dc.DeviceLayer(spec)
    wf = torch.empty_like(lay.weight)
    bf = torch.empty(c_out, device="cuda")
    dc.fold_bn(lay, wf, bf)
    packed = torch.empty(dc.packed_bytes(g, dc.BF16), dtype=torch.uint8, device="cuda")
    dc.pack_weights(wf, g, dc.BF16, packed)
    x = I.make_input(12, (n, h, w, c_in), bf16=True)
    ho, wo = O.out_extent(h, k, s, p), O.out_extent(w, k, s, p)
    r = I.round_bf16(I.normal(13, 99, (n, ho, wo, c_out)))
    Wf, bfo = O.fold_bn(spec)
    lin = O.conv_direct(x.transpose(0, 3, 1, 2), Wf, bfo, k, s, p)
    # plain, and with skip input + ReLU6
    y = run_conv(dc, dev(x, torch.bfloat16), g, packed, bf, dc.ACT_IDENTITY, algo=algo)
    assert_close(nchw(y), lin, TOL_BF16)
    y = run_conv(dc, dev(x, torch.bfloat16), g, packed, bf, dc.ACT_RELU6, residual=dev(r, torch.bfloat16), algo=algo)
    assert_close(nchw(y), O.relu6(lin + r.transpose(0, 3, 1, 2)), TOL_BF16)


@pytest.mark.parametrize("c_in,c_out,k,p,n,h,w", [
    (40, 16, 1, 0, 1, 3, 5),         # the fewest channels and fewer pixels than a block has rows
    (144, 24, 1, 0, 3, 37, 41),      # 24 outputs of 32 operand rows, ragged runs of pixels
    (520, 24, 1, 0, 5, 7, 7),        # a last plane of one chunk
    (64, 16, 3, 1, 2, 12, 70),       # one plane, column strips
    (40, 8, 3, 0, 1, 18, 41),        # eight outputs, no padding
    (112, 16, 3, 1, 104, 9, 9),      # several images
    (280, 16, 3, 2, 1, 14, 15),      # the widest padding, a long reduction of few items
    (40, 24, 5, 2, 1, 22, 300),      # wider than the fold kernel took
    (64, 8, 5, 4, 2, 9, 11),
    (136, 24, 5, 2, 1, 20, 66),
    (48, 24, 7, 3, 2, 15, 20),
    (72, 8, 7, 0, 1, 7, 9),          # one row of outputs
])
def test_narrow_outputs_by_rows_against_the_oracle(dc, c_in, c_out, k, p, n, h, w):
    test_each_forward_kernel_against_the_oracle(dc, c_in, c_out, k, 1, p, n, h, w, "k_conv_tc_rows")


@pytest.mark.parametrize("c_in,c_out,p,n,h,w,kernel", [
    (24, 8, 3, 2, 14, 14, "k_conv_tc_fold"),
    (24, 8, 0, 1, 7, 9, "k_conv_tc_fold"),           # one row of outputs
    (24, 8, 6, 1, 9, 300, "k_conv_tc_fold"),         # the widest padding, column strips
    (24, 16, 3, 1, 7, 8, "k_conv_tc_rows"),          # a plane of three chunks, fewer pixels than a block has rows
    (24, 16, 3, 1, 20, 260, "k_conv_tc_rows"),
    (24, 24, 3, 16, 28, 28, "k_conv_tc_rows"),       # 24 outputs of 32 operand rows
    (24, 24, 0, 3, 33, 41, "k_conv_tc_rows"),
    (32, 8, 2, 2, 15, 70, "k_conv_tc_rows"),
    (32, 16, 6, 5, 9, 11, "k_conv_tc_rows"),
    (32, 24, 3, 2, 14, 14, "k_conv_tc"),             # weights beyond the line for either
])
def test_7x7_of_few_channels_to_few_against_the_oracle(dc, c_in, c_out, p, n, h, w, kernel):
    test_each_forward_kernel_against_the_oracle(dc, c_in, c_out, 7, 1, p, n, h, w, kernel)


@pytest.mark.parametrize("c_in,c_out", [(24, 8), (24, 16), (24, 24), (32, 8)])
def test_three_3x3_layers_to_few_outputs_in_the_packed_order(dc, c_in, c_out):
    _check_delivery(dc, [I.make_layer(95, 0, c_in, 24, 3, 1, 1), I.make_layer(95, 1, 24, 40, 3, 1, 1), I.make_layer(95, 2, 40, c_out, 3, 1, 1)], [],
                    (dc.BF16, dc.F32))


@pytest.mark.parametrize("c_in,c_out,k,s,p,n,h,w,kernel", [
    (24, 24, 3, 1, 1, 3, 31, 23, "k_conv_tc_pairrows"),     # odd padding: the last pixel is the second of its output pair
    (32, 32, 5, 1, 2, 2, 28, 29, "k_conv_tc_pairrows"),     # even padding: the last output pair has one pixel
    (32, 32, 3, 1, 1, 51, 25, 25, "k_conv_tc_pairrows"),    # several tiles per CTA: more tiles than stages
    (16, 8, 3, 1, 0, 2, 18, 41, "k_conv_tc_pairrows"),      # no padding
    (8, 16, 3, 1, 1, 1, 6, 301, "k_conv_tc_pairrows"),      # three column strips: only the last one holds the column
    (16, 16, 7, 1, 3, 3, 20, 21, "k_conv_tc_pairrows"),     # 7x7
    (8, 8, 3, 1, 1, 200, 5, 3, "k_conv_tc_pairrows"),       # one whole pair per row
    (24, 24, 3, 1, 1, 1, 7, 7, "k_conv_tc_pairrows"),       # fewer outputs than a block has rows
    (16, 16, 5, 1, 2, 1, 1, 3, "k_conv_tc_pairrows"),       # the smallest odd width the map has a pair in
    (32, 16, 1, 1, 0, 2, 33, 25, "k_conv_tc_pairrows"),     # 1x1
    (16, 128, 3, 1, 1, 3, 12, 17, "k_conv_tc_pairrows"),    # two accumulator slots, run-time channel loop
    (24, 32, 3, 2, 1, 3, 28, 29, "k_conv_tc_pairrows"),     # stride 2: the column in both row planes
    (32, 16, 5, 2, 2, 2, 31, 45, "k_conv_tc_pairrows"),     # stride 2, even padding
    (16, 24, 3, 2, 0, 4, 17, 37, "k_conv_tc_pairrows"),     # stride 2, no padding
    (40, 32, 3, 2, 1, 2, 28, 29, "k_conv_tc_rows_s2"),       # stride 2 by sub-tiles
    (96, 144, 5, 2, 2, 1, 57, 57, "k_conv_tc_rows_s2"),      # the same, several tiles per image
    (24, 168, 3, 2, 1, 1, 49, 49, "k_conv_tc_rows_s2"),      # few channels, more outputs than the pair rows take
])
def test_odd_widths_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w, kernel):
    test_each_forward_kernel_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w, kernel)


@pytest.mark.parametrize("c_in,c_out,k,s,p,n,h,w", [
    (24, 24, 3, 1, 1, 1, 9, 15),         # pair rows
    (24, 32, 3, 2, 1, 2, 13, 11),        # pair rows, stride 2
    (48, 24, 3, 1, 1, 1, 10, 13),        # fold
    (72, 200, 3, 1, 1, 1, 7, 9),         # rows, two passes, a partial last plane
    (40, 264, 3, 2, 1, 1, 9, 13),        # rows, stride 2, two passes
    (32, 40, 1, 1, 0, 1, 9, 7),          # general
    (8, 136, 5, 2, 1, 1, 11, 13),        # general, stride 2
    (20, 12, 3, 1, 1, 1, 9, 7),          # channels no multiple of 8
])
def test_cuda_core_kernel_reads_every_weight_order(dc, c_in, c_out, k, s, p, n, h, w):
    test_each_forward_kernel_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w, None, algo=dc.ALGO_SIMT)


BIAS_CASES = [
    (32, 32, 3, 1, 1, 2, 9, 15),         # pair rows, odd width
    (24, 24, 3, 1, 1, 2, 10, 16),        # pair rows, even width
    (24, 32, 3, 2, 1, 2, 13, 11),        # pair rows, stride 2
    (144, 32, 3, 1, 1, 8, 28, 28),       # rows, resident weights
    (384, 64, 3, 1, 1, 1, 14, 14),       # rows, a shared reduction
    (128, 128, 5, 1, 2, 4, 30, 33),      # rows, 128 outputs of a 5x5 kernel
    (40, 32, 3, 2, 1, 2, 28, 29),        # rows, stride 2
    (48, 24, 3, 1, 1, 1, 20, 20),        # fold
    (200, 24, 3, 1, 1, 1, 14, 14),       # general
    (8, 136, 3, 2, 1, 1, 13, 15),        # general, stride 2
]


@pytest.mark.parametrize("c_in,c_out,k,s,p,n,h,w", BIAS_CASES)
def test_bias_keeps_its_32_bits(dc, c_in, c_out, k, s, p, n, h, w):
    """A bias that the products cancel down to its last 8 bits: y = b - hi - mid with hi and mid the two bf16 values that
    hold its first 16.  A few roundings of an fp32 sum are at most 2^-21 |b|; a bias held as two bf16 terms is off by 2^-17."""
    gen = torch.Generator().manual_seed(17)
    b = (torch.randn(c_out, generator=gen) * 2.0 ** torch.randint(-6, 7, (c_out,), generator=gen)).float()
    cut = lambda v: (v.view(torch.int32) & -65536).view(torch.float32)
    hi = cut(b)
    mid = cut(b - hi)
    w4 = torch.zeros(c_out, c_in, k, k)
    w4[:, 0, p, p], w4[:, 1, p, p] = -hi, -mid           # the centre tap: inside the image for every output
    x = torch.zeros(n, h, w, c_in)
    x[..., :2] = 1.0
    want = (b.double() - hi.double() - mid.double()).expand(n, *[O.out_extent(e, k, s, p) for e in (h, w)], c_out)
    g = dc.geom(c_in, c_out, 1, k, s, p)
    packed = torch.empty(dc.packed_bytes(g, dc.BF16), dtype=torch.uint8, device="cuda")
    dc.pack_weights(w4.cuda(), g, dc.BF16, packed)
    for algo in (dc.ALGO_AUTO, dc.ALGO_SIMT):
        y = run_conv(dc, x.cuda().bfloat16(), g, packed, b.cuda(), dc.ACT_IDENTITY, algo=algo).double().cpu()
        assert float(((y - want).abs() / b.double().abs()).max()) <= 2.0 ** -21


@pytest.mark.parametrize("c_in,c_out,k,s,p,n,h,w", BIAS_CASES)
def test_bias_that_is_not_finite(dc, c_in, c_out, k, s, p, n, h, w):
    """Infinities and NaN in the bias, and a finite value that rounds to a bf16 infinity, come out as from the CUDA-core
    kernel, and only in their own channels."""
    b = torch.linspace(-1, 1, c_out)
    b[:4] = torch.tensor([float("inf"), -float("inf"), float("nan"), 3.4e38])
    g = dc.geom(c_in, c_out, 1, k, s, p)
    packed = torch.empty(dc.packed_bytes(g, dc.BF16), dtype=torch.uint8, device="cuda")
    dc.pack_weights(torch.zeros(c_out, c_in, k, k).cuda(), g, dc.BF16, packed)
    x, ws = torch.ones(n, h, w, c_in, device="cuda", dtype=torch.bfloat16), torch.zeros(dc.conv_workspace_bytes(), dtype=torch.uint8, device="cuda")
    out = []
    for algo in (dc.ALGO_AUTO, dc.ALGO_SIMT):
        y = torch.empty(n, O.out_extent(h, k, s, p), O.out_extent(w, k, s, p), c_out, device="cuda", dtype=torch.bfloat16)
        dc.conv_forward(x, g, packed, b.cuda(), dc.ACT_IDENTITY, None, y, ws, algo=algo)
        assert dc.workspace_status(ws) == dc.OK
        out.append(y.float())
    assert torch.equal(torch.nan_to_num(out[0], nan=7e7), torch.nan_to_num(out[1], nan=7e7))
    assert bool(out[0][..., 2].isnan().all()) and not bool(out[0][..., 3:].isnan().any())
    # ReLU6 clamps them: a NaN becomes 0 in every kernel
    for algo in (dc.ALGO_AUTO, dc.ALGO_SIMT):
        dc.conv_forward(x, g, packed, b.cuda(), dc.ACT_RELU6, None, y, ws, algo=algo)
        assert [float(v) for v in y[..., :4].float().amax((0, 1, 2))] == [6.0, 0.0, 0.0, 6.0]
        assert [float(v) for v in y[..., :4].float().amin((0, 1, 2))] == [6.0, 0.0, 0.0, 6.0]


@pytest.mark.parametrize("c_in,c_out,k,s,p,n,h,w", [
    (128, 128, 5, 1, 2, 4, 30, 33),      # narrow strips whose whole steps fit, a shared reduction
    (72, 200, 5, 1, 2, 2, 11, 13),       # 5x5 in two passes, a partial plane of channels, a shared reduction
    (64, 200, 5, 1, 2, 24, 28, 28),      # two passes, more items than CTAs
    (16, 200, 7, 1, 3, 16, 30, 30),      # 16 channels, 7x7: whole steps of a quarter of a full plane's weights
    (72, 128, 5, 1, 2, 12, 50, 50),      # weight stages of one tap column, more items than CTAs
    (128, 256, 5, 1, 2, 6, 28, 28),      # the same in two passes, a shared reduction
    (48, 136, 7, 1, 3, 4, 26, 31),       # 48 channels, 7x7: two passes, runs cut by blocks
    (40, 48, 7, 1, 3, 1, 16, 40),        # 7x7
    (64, 64, 3, 1, 1, 2, 9, 120),        # wide rows: strips of 20 columns, whole height
    (64, 64, 3, 1, 1, 40, 5, 5),         # several small images per tile
    (64, 64, 1, 1, 0, 1, 3, 5),          # 1x1: one short run of pixels
    (96, 576, 1, 1, 0, 3, 13, 13),       # 1x1: pixels of several images in a tile, a ragged last tile
    (64, 384, 1, 1, 0, 64, 14, 14),      # 1x1: more tiles than CTAs
    (32, 96, 1, 1, 0, 1, 1, 1),          # one pixel
    (64, 128, 5, 1, 2, 1, 6, 1300),      # wide: the strips the tensor map allows do not fit beside the weights
    (128, 128, 7, 1, 3, 1, 8, 640),      # the same with 7x7
])
def test_rows_tiles_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w):
    test_each_forward_kernel_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w, "k_conv_tc_rows")


@pytest.mark.parametrize("c_in,c_out,k,s,p,n,h,w", [
    (160, 136, 3, 1, 1, 131, 7, 7),      # four images per tile, a ragged last group
    (64, 64, 5, 1, 2, 150, 5, 5),        # too little to save: not shared
    (72, 48, 7, 1, 3, 151, 4, 6),        # halo of three: as wide as half a map; the reduction shared as well
    (48, 144, 3, 1, 1, 153, 1, 3),       # not shared
    (64, 64, 3, 1, 2, 150, 6, 6),        # padding that is not half the kernel: nothing is shared
    (96, 64, 3, 1, 1, 40, 28, 28),       # not shared
    (40, 48, 3, 1, 1, 88, 17, 6),        # several images, ...
    (40, 104, 3, 1, 1, 75, 10, 10),      # ... with resident weights, ...
    (152, 64, 3, 1, 1, 32, 1, 36),       # ... of one row, the reduction shared
    (40, 56, 3, 1, 1, 15, 31, 31),       # whole rows of one image: halo columns only, ...
    (48, 96, 3, 1, 1, 22, 27, 27),       # ... with resident weights
    (40, 144, 5, 1, 2, 107, 1, 24),      # halo of two: one-row maps, every row between two images is halo, ...
    (48, 128, 5, 1, 2, 181, 2, 37),      # ... with weights by tap columns, ...
    (64, 184, 5, 1, 2, 11, 25, 25),      # ... the same with rows of one image, ...
    (80, 48, 5, 1, 2, 17, 23, 8),        # ... and with the reduction shared
    (56, 192, 7, 1, 3, 203, 2, 2),       # halo of three: wider than the map, ...
    (56, 144, 7, 1, 3, 230, 4, 4),       # ... as wide as most of it, weights by tap columns, ...
    (40, 72, 7, 1, 3, 29, 22, 22),       # ... and whole rows of one image
    (176, 88, 3, 1, 1, 16, 63, 63),      # wide maps, where whole rows are not the best tiles
    (160, 144, 3, 1, 1, 2, 106, 106),
    (144, 144, 5, 1, 2, 3, 41, 41),
])
def test_rows_with_shared_halos_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w):
    test_each_forward_kernel_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w, "k_conv_tc_rows")


@pytest.mark.parametrize("c_in,c_out,k,s,p,n,h,w", [
    (384, 64, 3, 1, 1, 1, 14, 14),       # one item for the chip: its 18 steps over a cluster of eight
    (960, 160, 1, 1, 0, 1, 7, 7),        # 1x1: 15 planes over a cluster
    (576, 200, 3, 1, 1, 2, 13, 9),       # several items, two passes, a ragged map
    (256, 128, 5, 1, 2, 1, 20, 21),      # weight stages of one tap column
    (160, 48, 3, 1, 1, 3, 5, 5),         # a half-filled last plane, several images per item
    (80, 32, 3, 1, 1, 1, 3, 4),          # fewer pixels than one warp reads
])
def test_rows_with_a_shared_reduction_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w):
    test_each_forward_kernel_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w, "k_conv_tc_rows")


@pytest.mark.parametrize("c_in,c_out,k,s,p,n,h,w", [
    (960, 1280, 1, 1, 0, 1, 7, 7),       # passes of the widest tile: most sums to read, one block
    (960, 1280, 1, 1, 0, 2, 15, 13),     # two blocks
    (320, 40, 1, 1, 0, 2, 30, 29),       # five planes, a ragged last tile
    (272, 328, 1, 1, 0, 2, 5, 5),        # a last pass with fewer channels than the tile, a plane of 16
    (128, 64, 3, 1, 1, 20, 13, 13),      # few steps, many items
    (1024, 40, 1, 1, 0, 1, 3, 3),        # few outputs: most threads have nothing to add
    (720, 72, 5, 1, 2, 1, 9, 31),        # the rings go round several times
])
def test_shared_reductions_of_few_and_many_sums(dc, c_in, c_out, k, s, p, n, h, w):
    test_each_forward_kernel_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w, "k_conv_tc_rows")


@pytest.mark.parametrize("c_in,c_out,k,s,p,n,h,w", [
    (96, 144, 5, 2, 2, 9, 57, 50),       # several tiles per image and per CTA, odd height
    (96, 144, 5, 2, 2, 1, 20, 20),       # the reduction shared by a cluster
    (64, 696, 3, 2, 1, 2, 12, 7),        # the same with one plane: CTAs with one or two of its six steps
    (72, 216, 3, 2, 1, 20, 17, 12),      # the same with two planes, the second of eight channels
    (40, 32, 3, 2, 1, 40, 28, 28),       # one image per tile, runs cut by blocks
    (40, 48, 3, 2, 1, 160, 21, 21),      # weights resident, more items than CTAs
    (48, 64, 7, 2, 3, 2, 31, 44),        # 7x7: classes of 16, 12, 12 and 9 taps
    (72, 200, 3, 2, 0, 1, 17, 150),      # no padding, column strips, a partial last plane
    (64, 264, 3, 2, 1, 2, 21, 19),       # two passes
    (160, 256, 5, 2, 1, 3, 15, 9),       # padding 1, 256 outputs: weight stages of one tap
    (24, 168, 3, 2, 1, 30, 9, 9),        # few channels, several images per tile
    (384, 24, 3, 2, 1, 1, 7, 7),         # few outputs
])
def test_stride_2_by_sub_tiles_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w):
    test_each_forward_kernel_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w, "k_conv_tc_rows_s2")


@pytest.mark.parametrize("c_in,c_out,k,s,p,n,h,w", [
    (8, 136, 3, 2, 1, 2, 28, 28),        # even width
    (8, 136, 3, 2, 1, 3, 27, 29),        # odd sides: the last column is in one parity plane only
    (8, 144, 5, 2, 2, 2, 22, 25),        # 5x5, even padding
    (8, 136, 5, 2, 1, 1, 31, 26),        # 5x5, odd tap columns lead
    (8, 200, 3, 2, 0, 1, 17, 151),       # no padding, two column strips
    (8, 264, 3, 2, 1, 2, 15, 13),        # two passes
])
def test_stride_2_on_parity_planes_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w):
    test_each_forward_kernel_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w, "k_conv_tc")


@pytest.mark.parametrize("c_in,c_out,k,s,p,n,h,w", [
    (32, 32, 5, 1, 2, 3, 28, 28),       # whole pixel tiles and a ragged last one
    (8, 40, 3, 1, 1, 1, 7, 9),          # a K slice of 16 spans two taps; 40 channels per tile
    (4, 20, 3, 2, 1, 2, 9, 11),         # four taps per slice, K no multiple of a slice, stride 2
    (12, 33, 5, 1, 2, 1, 8, 8),         # ragged taps in a slice, channels no multiple of 8
    (960, 160, 1, 1, 0, 1, 7, 7),       # K split over a cluster
    (160, 320, 3, 1, 1, 1, 7, 7),       # the same with taps
    (72, 16, 3, 1, 1, 1, 5, 5),         # a split whose last CTAs have fewer slices
    (24, 24, 7, 1, 3, 1, 9, 9),
    (16, 16, 1, 1, 0, 1, 1, 1),         # one pixel, one slice
    (64, 72, 3, 2, 0, 1, 15, 17),       # stride 2, no padding
    (40, 48, 3, 1, 1, 40, 25, 25),      # many tiles, none split
    (6, 8, 3, 1, 1, 2, 9, 9),           # channels no multiple of 4: the kernel that takes any count
])
def test_dense_fp32_against_the_oracle(dc, c_in, c_out, k, s, p, n, h, w):
    g = dc.geom(c_in, c_out, 1, k, s, p)
    spec = I.make_layer(14, 0, c_in, c_out, k, s, p)
    lay = dc.DeviceLayer(spec)
    wf = torch.empty_like(lay.weight)
    bf = torch.empty(c_out, device="cuda")
    dc.fold_bn(lay, wf, bf)
    packed = torch.empty(dc.packed_bytes(g, dc.F32), dtype=torch.uint8, device="cuda")
    dc.pack_weights(wf, g, dc.F32, packed)
    x = I.make_input(15, (n, h, w, c_in))
    ho, wo = O.out_extent(h, k, s, p), O.out_extent(w, k, s, p)
    r = I.normal(16, 99, (n, ho, wo, c_out))
    Wf, bfo = O.fold_bn(spec)
    lin = O.conv_direct(x.transpose(0, 3, 1, 2), Wf, bfo, k, s, p)
    # fp32 sums of up to 1440 products: errors of about 1e-6 of the result's rms, a hundredth of the bounds
    y = run_conv(dc, dev(x), g, packed, bf, dc.ACT_IDENTITY)
    assert_close(nchw(y), lin, TOL_F32, bf16=False)
    y = run_conv(dc, dev(x), g, packed, bf, dc.ACT_RELU6, residual=dev(r))
    assert_close(nchw(y), O.relu6(lin + r.transpose(0, 3, 1, 2)), TOL_F32, bf16=False)
    again = run_conv(dc, dev(x), g, packed, bf, dc.ACT_RELU6, residual=dev(r))
    assert torch.equal(y, again)


@pytest.mark.parametrize("c,k,s,p,n,h,w", [(64, 3, 1, 1, 2, 19, 21), (48, 3, 2, 1, 1, 20, 30), (32, 5, 1, 2, 1, 11, 13)])
def test_dwconv_stencil_without_activation(dc, c, k, s, p, n, h, w):
    """The stencil's instantiations without ReLU6 (tile widths 32 and 16, widths that are no multiple of a
    thread's item): negative and large outputs must come through unclamped."""
    spec = I.make_layer(18, 0, c, c, k, s, p, depthwise=True)
    lay = dc.DeviceLayer(spec)
    wf = torch.empty_like(lay.weight)
    bf = torch.empty(c, device="cuda")
    dc.fold_bn(lay, wf, bf)
    g = dc.geom(c, c, c, k, s, p)
    packed = torch.empty(dc.packed_bytes(g, dc.F32) // 4, dtype=torch.float32, device="cuda")
    dc.pack_weights(wf, g, dc.F32, packed)
    x = 4.0 * I.make_input(19, (n, h, w, c), bf16=True)
    x = I.round_bf16(x)
    ho, wo = O.out_extent(h, k, s, p), O.out_extent(w, k, s, p)
    gy = Guarded(torch, (n, ho, wo, c), torch.bfloat16, fill=float("nan"))
    dc.dwconv_forward(dev(x, torch.bfloat16), k, s, p, packed, bf, dc.ACT_IDENTITY, gy.t)
    assert dc.dwconv_status() == dc.OK
    gy.check("depthwise output")
    Wf, bfo = O.fold_bn(spec)
    ref = O.conv_direct(x.transpose(0, 3, 1, 2), Wf, bfo, k, s, p, groups=c)
    assert ref.min() < -1.0 and ref.max() > 6.5        # the case does exercise what ReLU6 would have cut
    assert_close(nchw(gy.t), ref, TOL_BF16, bf16=True)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("c,k,s,p,n,h,w", [(32, 3, 1, 1, 2, 12, 12), (96, 3, 2, 1, 1, 15, 17),
                                           (144, 3, 1, 1, 1, 9, 30), (20, 5, 1, 2, 1, 8, 8),
                                           (6, 3, 2, 1, 2, 7, 7), (960, 3, 1, 1, 2, 7, 7),
                                           # the shared-memory stencil: several row tiles with a ragged last one,
                                           # stride 2 with an odd height, 5x5 both strides, several images per tile
                                           (32, 3, 1, 1, 3, 150, 112), (96, 3, 2, 1, 2, 41, 112), (240, 5, 2, 2, 2, 28, 28),
                                           (384, 3, 1, 1, 21, 14, 14), (576, 5, 1, 2, 3, 14, 14), (24, 3, 1, 0, 2, 9, 20)])
def test_dwconv(dc, dtype, c, k, s, p, n, h, w):
    spec = I.make_layer(8, 0, c, c, k, s, p, depthwise=True)
    lay = dc.DeviceLayer(spec)
    wf = torch.empty_like(lay.weight)
    bf = torch.empty(c, device="cuda")
    dc.fold_bn(lay, wf, bf)
    g = dc.geom(c, c, c, k, s, p)
    packed = torch.empty(dc.packed_bytes(g, dc.F32) // 4, dtype=torch.float32, device="cuda")
    dc.pack_weights(wf, g, dc.F32, packed)
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    x = I.make_input(9, (n, h, w, c), bf16=(dtype == "bf16"))
    ho, wo = O.out_extent(h, k, s, p), O.out_extent(w, k, s, p)
    gy = Guarded(torch, (n, ho, wo, c), tdt, fill=float("nan"))
    y = gy.t
    dc.dwconv_forward(dev(x, tdt), k, s, p, packed, bf, dc.ACT_RELU6, y)
    assert dc.dwconv_status() == dc.OK
    gy.check("depthwise output")
    Wf, bfo = O.fold_bn(spec)
    ref = O.relu6(O.conv_direct(x.transpose(0, 3, 1, 2), Wf, bfo, k, s, p, groups=c))
    assert_close(nchw(y), ref, TOL_F32 if dtype == "f32" else TOL_BF16, bf16=(dtype == "bf16"))


@pytest.mark.parametrize("c,k,s,p,n,h,w", [
    (40, 3, 1, 1, 2, 9, 9),              # small maps: tiles of eight channels and a row
    (72, 3, 2, 1, 3, 15, 13),
    (8, 5, 1, 2, 1, 7, 7),
    (152, 3, 1, 1, 1, 27, 24),
    (104, 5, 2, 2, 9, 21, 23),
    (360, 3, 1, 1, 70, 7, 7),            # two rows per thread of an odd height, several images per tile
    (48, 3, 1, 1, 32, 56, 56),           # two rows per thread, more tiles than CTAs at once
    (8, 5, 2, 2, 1, 6, 252),             # widest maps of the load unit's box: the last items read past their row
    (16, 3, 1, 1, 1, 5, 254),
    (24, 3, 1, 1, 20, 12, 254),
    # one row per thread: tiles of 16 and 32 channels, the last one partly filled, several images in some
    (440, 3, 1, 1, 21, 6, 3), (360, 3, 1, 1, 38, 4, 4), (480, 3, 1, 1, 39, 3, 3), (152, 3, 2, 1, 25, 5, 11), (152, 3, 2, 1, 47, 3, 3),
    (440, 5, 1, 2, 21, 4, 9), (408, 5, 2, 2, 21, 3, 3), (432, 5, 2, 2, 21, 6, 6),
    # two rows per thread, odd heights: the same
    (456, 3, 1, 1, 22, 5, 3), (176, 3, 1, 1, 28, 9, 8), (216, 3, 1, 1, 125, 3, 3), (40, 3, 2, 1, 62, 17, 17), (280, 3, 2, 1, 71, 5, 3),
    (272, 5, 1, 2, 35, 6, 3), (104, 5, 1, 2, 23, 11, 11), (440, 5, 1, 2, 124, 5, 3), (440, 5, 2, 2, 11, 9, 9), (264, 5, 2, 2, 71, 6, 3),
])
def test_dwconv_stencil_tiles(dc, c, k, s, p, n, h, w):
    test_dwconv_stencil_without_activation(dc, c, k, s, p, n, h, w)
    test_dwconv(dc, "bf16", c, k, s, p, n, h, w)


@pytest.mark.parametrize("c,k,w,becomes", [(16, 3, 9, 6.0), (40, 5, 9, 6.0), (16, 3, 300, 0.0), (12, 3, 9, 0.0), (16, 7, 9, 0.0)])
def test_relu6_of_a_nan_in_depthwise_layers(dc, c, k, w, becomes):
    """6 in the stencil, 0 in the kernels for what it does not take: wider maps, other channel counts, other kernel sizes."""
    g = dc.geom(c, c, c, k, 1, k // 2)
    packed = torch.empty(dc.packed_bytes(g, dc.F32), dtype=torch.uint8, device="cuda")
    dc.pack_weights(torch.zeros(c, 1, k, k, device="cuda"), g, dc.F32, packed)
    b = torch.ones(c, device="cuda")
    b[1] = float("nan")
    x, y = torch.zeros(2, 5, w, c, dtype=torch.bfloat16, device="cuda"), torch.empty(2, 5, w, c, dtype=torch.bfloat16, device="cuda")
    dc.dwconv_forward(x, k, 1, k // 2, packed, b, dc.ACT_RELU6, y)
    assert dc.dwconv_status() == dc.OK
    assert bool((y[..., 1] == becomes).all()) and bool((y[..., 2:] == 1).all())


@pytest.mark.parametrize("c_in,hidden,c_out,s,n,h,w,biases,one_launch", [
    (16, 96, 16, 1, 3, 9, 11, True, True),       # two groups of warps, a ragged map
    (64, 384, 64, 1, 5, 14, 14, True, True),     # six chunks of 64 hidden channels
    (40, 240, 232, 2, 1, 25, 26, True, True),    # stride 2, odd height, two passes of output channels
    (24, 80, 32, 1, 2, 13, 12, False, True),     # chunks of 48 and 32, no biases
    (24, 96, 8, 1, 2, 13, 12, True, True),       # eight outputs
    (24, 80, 8, 1, 2, 13, 12, True, False),      # projection weights in groups of five chunks, padded to six: three launches
    (72, 432, 40, 1, 1, 33, 34, True, True),     # a last pass of hidden channels that is shorter than the others
    (16, 96, 24, 2, 1, 40, 112, True, True),     # several strips of columns
    (24, 144, 24, 1, 40, 20, 20, True, True),    # tiles of 7 columns, three strips to an image
    (32, 192, 32, 1, 77, 10, 10, False, True),   # a tile to each image
    (40, 240, 40, 1, 64, 20, 20, True, True),    # two groups of warps, one buffer for the projection's operand
    (16, 96, 264, 1, 1, 12, 12, True, False),    # more than 256 outputs: three launches
    (24, 72, 24, 1, 1, 12, 12, True, False),     # hidden channels no multiple of 16: three launches
])
def test_block_in_one_launch_against_the_oracle(dc, c_in, hidden, c_out, s, n, h, w, biases, one_launch):
    mk = I.make_layer
    specs = [mk(91, 0, c_in, hidden, 1, 1, 0, act="relu6", with_bn=False, with_bias=biases),
             mk(91, 1, hidden, hidden, 3, s, 1, depthwise=True, act="relu6", with_bn=False, with_bias=biases),
             mk(91, 2, hidden, c_out, 1, 1, 0, with_bn=False, with_bias=biases)]
    res = s == 1 and c_in == c_out
    keep, ptrs = [], []
    for spec, code in zip(specs, (dc.BF16, dc.F32, dc.BF16)):
        lay = dc.DeviceLayer(spec)
        g = dc.geom(spec.c_in, spec.c_out, spec.groups, spec.k, spec.stride, spec.pad)
        packed = torch.empty(dc.packed_bytes(g, code), dtype=torch.uint8, device="cuda")
        dc.pack_weights(lay.weight, g, code, packed)
        keep.append((lay, packed))
        ptrs += [packed.data_ptr(), lay.bias.data_ptr() if biases else None]
    blk = dc.Block(c_in, hidden, c_out, 1, 3, s, 1, int(res), dc.ACT_RELU6, dc.ACT_RELU6, *ptrs)
    x = I.make_input(92, (n, h, w, c_in), bf16=True)
    gy = Guarded(torch, (n, O.out_extent(h, 3, s, 1), O.out_extent(w, 3, s, 1), c_out), torch.bfloat16, fill=float("nan"))
    gws = Guarded(torch, (dc.block_workspace_bytes(n, h, w, blk, dc.BF16),), torch.uint8, fill=0)
    dc.block_forward(dev(x, torch.bfloat16), blk, gy.t, gws.t)
    assert dc.workspace_status(gws.t) == dc.OK
    gy.check("block output")
    gws.check("block workspace")
    assert (not bool(gws.t[256:].any())) == one_launch          # the hidden maps were never in the workspace
    assert (dc.block_plan(n, h, w, blk, dc.BF16) is not None) == one_launch
    cur = x.transpose(0, 3, 1, 2).astype(np.float64)
    skip = cur
    for spec in specs:
        Wf, bfo = O.fold_bn(spec)
        cur = O.conv_direct(cur, Wf, bfo, spec.k, spec.stride, spec.pad, spec.groups)
        cur = O.relu6(cur) if spec.act == "relu6" else cur
    assert_close(nchw(gy.t), cur + skip if res else cur, 3 * TOL_BF16, scale=3.0)      # as for three launches: the same roundings


# What a plan may have: form of the kernel (0 and 1: one group of warps), buffers of the projection's operand, weight stages, several
# images in a tile, several tiles for a CTA.
BLOCK_PLANS = [
    # c_in, hidden, c_out, s, n, h, w, (form, operands, stages, images, tiles)
    (24, 144, 24, 1, 40, 40, 40, (2, 1, 3, False, True)),
    (24, 144, 24, 1, 78, 15, 14, (2, 2, 3, False, True)),
    (16, 96, 16, 1, 76, 18, 18, (2, 2, 2, False, True)),
    (16, 96, 16, 2, 314, 13, 13, (2, 1, 2, True, True)),
    (24, 144, 24, 1, 300, 3, 3, (3, 2, 3, True, False)),
    (24, 144, 24, 1, 153, 11, 11, (3, 1, 3, True, False)),
    (24, 144, 24, 1, 83, 15, 15, (3, 2, 3, False, True)),
    (16, 240, 16, 1, 300, 16, 16, (3, 1, 4, False, True)),
    (16, 512, 16, 1, 82, 11, 11, (3, 2, 4, False, True)),
    (32, 192, 32, 1, 64, 28, 28, (0, 1, 2, False, False)),
    (24, 144, 24, 1, 75, 32, 32, (0, 1, 3, False, True)),
    (24, 144, 160, 1, 53, 17, 17, (0, 2, 3, False, False)),
    (16, 96, 24, 2, 20, 112, 112, (0, 2, 2, False, True)),
    (16, 96, 16, 1, 156, 12, 12, (1, 1, 2, True, False)),
    (16, 96, 16, 1, 21, 64, 64, (1, 1, 2, False, True)),
    (24, 144, 72, 1, 203, 11, 11, (1, 2, 3, True, False)),
    (16, 96, 8, 2, 125, 38, 34, (1, 2, 2, False, True)),
]


@pytest.mark.parametrize("c_in,hidden,c_out,s,n,h,w,plan", BLOCK_PLANS)
def test_block_plans_against_the_oracle(dc, c_in, hidden, c_out, s, n, h, w, plan):
    """Every form of the one-launch block kernel with what its loops carry from tile to tile and from image to image.  The plan is
    asked for, so that a change of the choice between plans cannot take a case from here unseen."""
    blk = dc.Block(c_in, hidden, c_out, 1, 3, s, 1, int(s == 1 and c_in == c_out), dc.ACT_RELU6, dc.ACT_RELU6, None, None, None, None, None, None)
    p = dc.block_plan(n, h, w, blk, dc.BF16)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert (p.form, p.operands, p.stages, p.tile_images > 1, p.tiles > sms) == plan
    test_block_in_one_launch_against_the_oracle(dc, c_in, hidden, c_out, s, n, h, w, True, True)


def test_block_in_place(dc):
    """An output on the block's own input goes through the workspace, and gives what a separate one gives."""
    n, h, w, c, m = 3, 14, 14, 24, 144
    gen = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda *shape: torch.randn(*shape, generator=gen, device="cuda")
    ptrs, keep = [], []
    for wt, (ci, co, groups, k), code in ((rnd(m, c, 1, 1) / c ** 0.5, (c, m, 1, 1), dc.BF16), (rnd(m, 1, 3, 3) / 3, (m, m, m, 3), dc.F32),
                                          (rnd(c, m, 1, 1) / m ** 0.5, (m, c, 1, 1), dc.BF16)):
        g = dc.geom(ci, co, groups, k, 1, k // 2)
        packed = torch.empty(dc.packed_bytes(g, code), dtype=torch.uint8, device="cuda")
        dc.pack_weights(wt, g, code, packed)
        keep += [packed, rnd(co)]
        ptrs += [packed.data_ptr(), keep[-1].data_ptr()]
    blk = dc.Block(c, m, c, 1, 3, 1, 1, 1, dc.ACT_RELU6, dc.ACT_RELU6, *ptrs)
    x = rnd(n, h, w, c).bfloat16()
    ws = torch.zeros(dc.block_workspace_bytes(n, h, w, blk, dc.BF16), dtype=torch.uint8, device="cuda")
    y = torch.empty_like(x)
    dc.block_forward(x, blk, y, ws)
    assert not bool(ws[256:].any())
    dc.block_forward(x, blk, x, ws)
    assert bool(ws[256:].any())
    assert torch.allclose(x.float(), y.float(), rtol=2.0 ** -7, atol=2.0 ** -6)      # one bf16 step, sums in another order


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("c_in,c_out,t,s,n,h,w", [(24, 24, 6, 1, 2, 14, 14), (16, 24, 6, 2, 1, 16, 16),
                                                  (32, 16, 1, 1, 1, 12, 12)])
def test_block_forward(dc, dtype, c_in, c_out, t, s, n, h, w):
    specs = I.inverted_residual(10, 0, c_in, c_out, t, s, block=0)
    code = dc.F32 if dtype == "f32" else dc.BF16
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    keep, packed, biases = [], [], []
    for spec in specs:
        lay = dc.DeviceLayer(spec)
        wf = torch.empty_like(lay.weight)
        bf = torch.empty(spec.c_out, device="cuda")
        dc.fold_bn(lay, wf, bf)
        g = dc.geom(spec.c_in, spec.c_out, spec.groups, spec.k, spec.stride, spec.pad)
        pk = torch.empty(dc.packed_bytes(g, code), dtype=torch.uint8, device="cuda")
        dc.pack_weights(wf, g, code, pk)
        packed.append(pk)
        biases.append(bf)
        keep.append((lay, wf))
    has_exp = t != 1
    res = s == 1 and c_in == c_out
    if has_exp:
        pe, pd, pp = packed
        be, bd, bp = biases
    else:
        (pd, pp), (bd, bp) = packed, biases
        pe = be = None
    blk = dc.Block(c_in, c_in * t, c_out, int(has_exp), 3, s, 1, int(res), dc.ACT_RELU6, dc.ACT_RELU6,
                   pe.data_ptr() if has_exp else None, be.data_ptr() if has_exp else None,
                   pd.data_ptr(), bd.data_ptr(), pp.data_ptr(), bp.data_ptr())
    x = I.make_input(11, (n, h, w, c_in), bf16=(dtype == "bf16"))
    ho = O.out_extent(h, 3, s, 1)
    wo = O.out_extent(w, 3, s, 1)
    gy = Guarded(torch, (n, ho, wo, c_out), tdt, fill=float("nan"))
    gws = Guarded(torch, (max(dc.block_workspace_bytes(n, h, w, blk, code), dc.conv_workspace_bytes()),), torch.uint8,
                  fill=0)
    y, ws = gy.t, gws.t
    dc.block_forward(dev(x, tdt), blk, y, ws)
    assert dc.workspace_status(ws) == dc.OK
    gy.check("block output")
    gws.check("block workspace")
    cur = x.transpose(0, 3, 1, 2).astype(np.float64)
    skip = cur
    for spec in specs:
        Wf, bfo = O.fold_bn(spec)
        cur = O.conv_direct(cur, Wf, bfo, spec.k, spec.stride, spec.pad, spec.groups)
        if spec.act == "relu6":
            cur = O.relu6(cur)
    if res:
        cur = cur + skip
    # bf16: three roundings of the intermediate maps on the GPU side -> 3x the single-layer budget
    if dtype == "f32":
        assert_close(nchw(y), cur, TOL_F32, bf16=False)
    else:
        assert_close(nchw(y), cur, 3 * TOL_BF16, scale=3.0)


@pytest.mark.parametrize("idx", [1, 2, 3])
def test_full_size_configs_on_every_image(dc, idx):
    """The batch-64/128 workloads in the launch configuration the benchmark times, every image
    against the oracle's sequential chain (each CTA owns a run of tiles somewhere in the batch, so a
    sample of images would leave most CTAs unchecked)."""
    case = I.chain_case(idx)
    g, wm, bm, packed = run_merge(dc, case.layers, case.residuals, packed_dtype=dc.BF16)
    W, b, k, s, p = O.merge_formula(case.layers, case.residuals)
    assert O.rel_l2(wm.cpu().numpy(), W) <= TOL_W and O.rel_l2(bm.cpu().numpy(), b) <= TOL_W
    x = case.x()
    y = run_conv(dc, dev(x, torch.bfloat16), g, packed, bm, dc.ACT_IDENTITY)
    ref = O.chain_forward_reordered(x.transpose(0, 3, 1, 2), case.layers, case.residuals)
    r, worst, max_abs = assert_close(nchw(y), ref, TOL_BF16, what=case.name)
    print("%s: rel-L2 %.3e, worst element at %.2f of its bound, max abs error %.3e" % (case.name, r, worst, max_abs))
    # per image as well: no single image may carry the whole error budget
    yn = nchw(y)
    for i in range(x.shape[0]):
        assert O.rel_l2(yn[i], ref[i]) <= TOL_BF16, (case.name, i)


def test_host_entry_point_matches_device_path(dc):
    case = I.chain_case(1, batch=4)
    arr, keep = dc.host_layer_array(case.layers)
    n, h, w, c = case.x_shape
    nbytes = dc.chain_host_workspace_bytes(arr, len(case.layers), case.residuals, n, h, w, dc.BF16)
    ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
    xh = torch.from_numpy(case.x()).to(torch.bfloat16).pin_memory()
    yh = torch.empty((n, h, w, 24), dtype=torch.bfloat16).pin_memory()
    dc.chain_forward_host(arr, len(case.layers), case.residuals, xh, dc.ACT_IDENTITY, yh, ws)
    assert dc.workspace_status(ws) == dc.OK
    ref = O.chain_forward_reordered(case.x().transpose(0, 3, 1, 2), case.layers, case.residuals)
    assert_close(yh.float().numpy().transpose(0, 3, 1, 2), ref, TOL_BF16)


def test_async_host_entry_point_overlaps_streams_and_matches_the_oracle(dc):
    # three batches in flight on three streams, each with its own workspace and pinned buffers
    arrs, outs, streams, cases = [], [], [], []
    for slot in range(3):
        case = I.chain_case(1, seed=20 + slot, batch=3)
        # slots 0 and 1: one pinned parameter block in the library's layout (a single transfer); slot 2: loose arrays
        arr, keep = dc.host_layer_array(case.layers, pinned=(slot < 2))
        n, h, w, c = case.x_shape
        nbytes = dc.chain_host_workspace_bytes(arr, len(case.layers), case.residuals, n, h, w, dc.BF16)
        ws = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
        xh = torch.from_numpy(case.x()).to(torch.bfloat16).pin_memory()
        yh = torch.zeros((n, h, w, 24), dtype=torch.bfloat16).pin_memory()
        st = torch.cuda.Stream()
        arrs.append((arr, keep, ws, xh))
        outs.append(yh); streams.append(st); cases.append(case)
    torch.cuda.synchronize()
    for slot in range(3):
        arr, keep, ws, xh = arrs[slot]
        dc.chain_forward_host_async(arr, len(cases[slot].layers), cases[slot].residuals, xh, dc.ACT_IDENTITY,
                                    outs[slot], ws, streams[slot])
    for slot in range(3):
        streams[slot].synchronize()
        assert dc.workspace_status(arrs[slot][2], streams[slot]) == dc.OK
        case = cases[slot]
        ref = O.chain_forward_reordered(case.x().transpose(0, 3, 1, 2), case.layers, case.residuals)
        assert_close(outs[slot].float().numpy().transpose(0, 3, 1, 2), ref, TOL_BF16)


def test_empty_and_degenerate_inputs_are_rejected_or_handled(dc):
    g = dc.geom(8, 8, 1, 3, 1, 1)
    packed = torch.zeros(dc.packed_bytes(g, dc.BF16), dtype=torch.uint8, device="cuda")
    x = torch.zeros((1, 1, 1, 8), dtype=torch.bfloat16, device="cuda")
    y = run_conv(dc, x, g, packed, None, dc.ACT_IDENTITY)            # 1x1 image, all taps but one in the padding
    assert y.shape == (1, 1, 1, 8) and float(y.float().abs().max()) == 0.0
    with pytest.raises(dc.DcError) as e:
        dc.conv_forward(torch.zeros((1, 2, 2, 8), dtype=torch.bfloat16, device="cuda"), dc.geom(8, 8, 1, 5, 1, 0),
                        packed, None, 0, None, y, new_ws(dc))
    assert e.value.status == dc.ERR_SHAPE


# n, h, w, c_in, c_out, k, stride, pad: runs of 256 and 128 lines, 16 to 80 outputs a tile, reductions shared by 2 to 8 CTAs, loads of
# rows, of several and of whole images, odd sides, odd channel groups, outputs that end inside a tile, both strides, more and less
# padding than "same", shallow rings
F32_TC_SHAPES = [(32, 28, 28, 32, 32, 5, 1, 2), (3, 52, 52, 48, 128, 3, 1, 1), (1, 44, 44, 192, 72, 5, 1, 2), (3, 97, 97, 160, 72, 3, 2, 1),
                 (2, 41, 43, 96, 112, 5, 2, 2), (78, 15, 15, 328, 56, 1, 1, 0), (20, 31, 31, 20, 36, 5, 1, 2), (2, 60, 60, 24, 24, 7, 1, 3),
                 (4, 61, 59, 64, 96, 3, 1, 0), (4, 61, 59, 64, 96, 3, 1, 2), (2, 33, 250, 64, 64, 3, 1, 1), (12, 43, 43, 64, 16, 5, 1, 2),
                 (40, 11, 11, 96, 96, 3, 1, 1), (1, 37, 37, 208, 72, 5, 1, 2), (2, 7, 7, 512, 512, 3, 1, 1), (8, 14, 14, 384, 64, 3, 1, 1)]


@pytest.mark.parametrize("shape", F32_TC_SHAPES)
def test_fp32_conv_by_bf16_terms(dc, shape):
    """fp32 on the tensor core against torch in 64 bits: at most as far from it as the FMA kernel (which the smaller shapes of this
    file hold to the oracle) and within 4e-7 of the result (2-norm; short sums of exact products, then fp32 additions of at most
    225 of them: 225 ** 0.5 * 2 ** -25), with bias, skip input and ReLU6 and without; guarded output; an infinity and a NaN in the
    input and in the weights come out as in the FMA kernel."""
    n, h, w, ci, co, k, s, p = shape
    g = dc.geom(ci, co, 1, k, s, p)
    assert dc.conv_kernel_name(n, h, w, g, dc.F32) == "k_conv_f32_tc"
    gen = torch.Generator("cuda")
    gen.manual_seed(ci * 1000 + co)
    rnd = lambda *d: torch.randn(d, generator=gen, device="cuda")
    x, wf = rnd(n, h, w, ci), rnd(co, ci, k, k) * (ci * k * k) ** -0.5
    ho, wo = (h + 2 * p - k) // s + 1, (w + 2 * p - k) // s + 1
    bias, res = rnd(co), rnd(n, ho, wo, co)
    packed = torch.empty(dc.packed_bytes(g, dc.F32), dtype=torch.uint8, device="cuda")
    dc.pack_weights(wf, g, dc.F32, packed)
    ws = torch.zeros(dc.conv_workspace_bytes(), dtype=torch.uint8, device="cuda")

    def run(algo, full=False):
        y = Guarded(torch, (n, ho, wo, co), torch.float32, fill=float("nan"))
        dc.conv_forward(x, g, packed, bias if full else None, dc.ACT_RELU6 if full else dc.ACT_IDENTITY, res if full else None, y.t, ws,
                        algo=algo)
        y.check("output")
        return y.t

    ref = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), wf.double(), None, s, p).permute(0, 2, 3, 1)
    err = lambda y, r: ((y.double() - r).norm() / r.norm()).item()
    worst = lambda y, r: ((y.double() - r).abs().max() / r.square().mean().sqrt()).item()
    y = run(dc.ALGO_AUTO)
    assert err(y, ref) <= min(4e-7, 1.02 * err(run(dc.ALGO_SIMT), ref)) and worst(y, ref) <= 1e-5
    full = (ref + bias.double() + res.double()).clamp(0, 6)
    y = run(dc.ALGO_AUTO, full=True)
    assert err(y, full) <= 4e-7 and worst(y, full) <= 1e-5
    assert dc.workspace_status(ws) == dc.OK
    # what is not finite
    x[0, 0, 0, 0], x[n - 1, h - 1, w - 1, ci - 1], x[0, h // 2, w // 2, ci // 2] = float("inf"), float("nan"), 3.4e38
    view = packed.view(torch.float32)[:k * k * ci * co].view(k, k, ci, co)
    view[k // 2, k // 2, ci - 1, 0], view[0, 0, 0, co - 1] = float("-inf"), float("nan")
    a, b = run(dc.ALGO_AUTO), run(dc.ALGO_SIMT)
    same = (a == b) | (torch.isnan(a) & torch.isnan(b))
    close = (a - b).abs() <= 1e-5 * b.abs().clamp(min=1.0)
    assert bool((same | (close & torch.isfinite(b))).all()) and bool((~torch.isfinite(b)).any())


@pytest.mark.parametrize("a,c,o,res,codes", [
    (104, 208, 136, [], "both"),               # a round of tiles and a bit
    (40, 120, 192, [], "both"),                # a tile a CTA, 8 of the last step's 64 channels
    (64, 200, 152, [], "both"),                # the same, a few tiles fewer than CTAs (the one above may go to the FMAs)
    (256, 256, 256, [], "both"),               # runs of tiles that change columns
    (196, 132, 250, [], "f32"),                # nothing a multiple of a tile or a step
    (168, 168, 168, [(0, 0)], "both"), (168, 168, 168, [(0, 0), (1, 1)], "both"), (168, 168, 168, [(0, 1)], "both"),
    (160, 320, 160, [], "both"),               # columns' terms cut again for every tile
    (24, 1216, 40, [], "both"),                # a packed order that holds pixels in its rows
])
def test_3x3_after_3x3_by_bf16_terms_against_the_oracle(dc, a, c, o, res, codes):
    specs = [I.make_layer(86, 0, a, c, 3, 1, 1), I.make_layer(86, 1, c, o, 3, 1, 1)]
    _check_delivery(dc, specs, res, (dc.BF16, dc.F32) if codes == "both" else (dc.F32,))
    assert dc.dwconv_status() == dc.OK
    if c >= 192 and not res:
        # sums of 128 products in the tensor core, cut below 2 ** -24 of the largest, then fp32 additions: 1.7e-7 measured at most; one
        # chain of FMAs over that many channels is 2.05e-7 or more away (so this also tells that it was not taken)
        W = O.merge_formula(specs, res)[0]
        _, wm, _, _ = run_merge(dc, specs, res, packed_dtype=dc.F32)
        assert O.rel_l2(wm.cpu().numpy(), W) <= 1.95e-7


@pytest.mark.parametrize("kind,a,c,o", [("33", 64, 136, 152), ("33", 256, 256, 256), ("33", 104, 208, 136), ("block", 160, 960, 160),
                                        ("block", 96, 576, 96), ("block", 200, 928, 200), ("pair", 320, 1280, 320), ("pair", 504, 504, 504)])
def test_merges_by_bf16_terms_of_weights_of_one_sign(dc, kind, a, c, o):
    """The tensor core cuts its sums, which adds up where all products have one sign: L steps of a sum lose (L + 1) / 2 x 2 ** -24 of it at
    0.7 on average over a binade, 1.1e-7 for the four of a 3x3 pair and 1.3e-7 for the five of the widest block here; beside the
    roundings of FMA kernels, 1e-7.  Weights of both signs: at most 1.7e-7 measured, and 3x3 pairs 1.3e-7 (1.85e-7 or more by FMAs)."""
    mk = I.make_layer
    if kind == "33":
        specs = [mk(97, 0, a, c, 3, 1, 1), mk(97, 1, c, o, 3, 1, 1)]
    else:
        specs = [mk(97, 0, a, c, 1, 1, 0), mk(97, 2, c, o, 1, 1, 0)]
        if kind == "block":
            specs.insert(1, mk(97, 1, c, c, 3, 1, 1, depthwise=True))
    for sign in (False, True):
        if sign:
            for s in specs:
                s.weight[...] = np.abs(s.weight)
        _, wm, _, _ = run_merge(dc, specs, [], packed_dtype=dc.F32)
        err = O.rel_l2(wm.cpu().numpy(), O.merge_formula(specs, [])[0])
        assert err <= (1.8e-7 if sign else 1.5e-7 if kind == "33" else 1.9e-7), (sign, err)


def test_3x3_after_3x3_by_bf16_terms_as_a_piece(dc):
    _check_delivery(dc, [I.make_layer(87, 0, 120, 200, 3, 1, 1), I.make_layer(87, 1, 200, 136, 3, 1, 1), I.make_layer(87, 2, 136, 16, 1, 1, 0)], [],
                    (dc.BF16, dc.F32))


@pytest.mark.parametrize("shape", F32_TC_SHAPES[:8])
def test_fp32_conv_by_bf16_terms_of_one_sign_and_of_small_values(dc, shape):
    """Maps behind ReLU6 under weights of one sign, where what the tensor core cuts off adds up: four steps of a sum lose 2.5 x 2 ** -24 x 0.7 =
    1e-7 of it at most, so no further from 64 bits than FMAs' 0.7e-7 or more by a tenth.  And values as small as terms reach: exact
    from 2 ** -110 on, below it to within 2 ** -133."""
    n, h, w, ci, co, k, s, p = shape
    g = dc.geom(ci, co, 1, k, s, p)
    assert dc.conv_kernel_name(n, h, w, g, dc.F32) == "k_conv_f32_tc"
    gen = torch.Generator("cuda")
    gen.manual_seed(ci * 1000 + co + 1)
    rnd = lambda *d: torch.randn(d, generator=gen, device="cuda")
    x, wf = rnd(n, h, w, ci), rnd(co, ci, k, k) * (ci * k * k) ** -0.5
    packed = torch.empty(dc.packed_bytes(g, dc.F32), dtype=torch.uint8, device="cuda")
    ws = torch.zeros(dc.conv_workspace_bytes(), dtype=torch.uint8, device="cuda")
    y = torch.empty((n, (h + 2 * p - k) // s + 1, (w + 2 * p - k) // s + 1, co), device="cuda")

    def err(x, wf, algo):
        dc.pack_weights(wf, g, dc.F32, packed)
        dc.conv_forward(x, g, packed, None, dc.ACT_IDENTITY, None, y, ws, algo=algo)
        ref = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), wf.double(), None, s, p).permute(0, 2, 3, 1)
        return ((y.double() - ref).norm() / ref.norm()).item()

    sign = (x * 2).clamp(0, 6), wf.abs()
    assert err(*sign, dc.ALGO_AUTO) <= min(1.2e-7, 1.1 * err(*sign, dc.ALGO_SIMT))
    assert err(x * 2.0 ** -104, wf * 2.0 ** 104, dc.ALGO_AUTO) <= 4e-7           # a thousandth of the values is below 2 ** -114
    assert err(x * 2.0 ** -120, wf * 2.0 ** 104, dc.ALGO_AUTO) <= 2.0 ** -13
    assert dc.workspace_status(ws) == dc.OK


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_fp32_conv_by_bf16_terms_of_maps_that_are_not_finite(dc, value):
    n, h, w, ci, co, k, s, p = F32_TC_SHAPES[0]
    g = dc.geom(ci, co, 1, k, s, p)
    x = torch.full((n, h, w, ci), value, device="cuda")
    x[1] = 1.0                                     # one image is
    wf = torch.full((co, ci, k, k), 0.5, device="cuda")
    wf[3] = -0.5
    packed = torch.empty(dc.packed_bytes(g, dc.F32), dtype=torch.uint8, device="cuda")
    dc.pack_weights(wf, g, dc.F32, packed)
    ws = torch.zeros(dc.conv_workspace_bytes(), dtype=torch.uint8, device="cuda")
    a, b = (torch.empty((n, h, w, co), device="cuda") for _ in range(2))
    dc.conv_forward(x, g, packed, None, dc.ACT_IDENTITY, None, a, ws)
    dc.conv_forward(x, g, packed, None, dc.ACT_IDENTITY, None, b, ws, algo=dc.ALGO_SIMT)
    assert torch.equal(a.nan_to_num(7.0), b.nan_to_num(7.0)) and bool(torch.isfinite(a[1]).all()) and not bool(torch.isfinite(a[0]).any())


def whole_numbers(seed, shape, top):
    return np.random.default_rng(seed).integers(-top, top + 1, shape).astype(np.float32)


@pytest.mark.parametrize("kind,a,c,o", [
    ("33", 256, 256, 256),                     # 3x3 pairs: up to five tiles a CTA, columns' terms that stay
    ("33", 320, 384, 256),                     # columns' terms cut again for every tile
    ("33", 168, 168, 168),                     # two tiles a CTA
    ("block", 160, 960, 160),                  # a slot's second use is the other team's step
    ("block", 200, 928, 200), ("block", 252, 700, 300), ("block", 96, 576, 96),
    ("pair", 960, 320, 1280), ("pair", 320, 1280, 320), ("pair", 72, 1500, 72),
])
def test_merges_by_bf16_terms_of_whole_numbers_are_exact_every_time(dc, kind, a, c, o):
    """Sums of whole numbers below 2 ** 24 are exact in any order, so one operand that a step reads too early, too late or from another
    step shows, however small its share.  Many runs, with other kernels between them."""
    mk = I.make_layer
    if kind == "33":
        specs = [mk(96, 0, a, c, 3, 1, 1, with_bn=False), mk(96, 1, c, o, 3, 1, 1, with_bn=False)]
    else:
        specs = [mk(96, 0, a, c, 1, 1, 0, with_bn=False), mk(96, 2, c, o, 1, 1, 0, with_bn=False)]
        if kind == "block":
            specs.insert(1, mk(96, 1, c, c, 3, 1, 1, depthwise=True, with_bn=False))
    for i, s in enumerate(specs):
        s.weight[...] = whole_numbers(a + i, s.weight.shape, 8)
    layers = [dc.DeviceLayer(s) for s in specs]
    g, ws_bytes = dc.merge_query(layers, [])
    wm, bm = torch.empty((g.c_out, g.c_in, g.k, g.k), device="cuda"), torch.empty(g.c_out, device="cuda")
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device="cuda")
    w1, w2 = layers[0].weight.double(), layers[-1].weight.double()
    if kind == "33":
        ref = torch.zeros(wm.shape, dtype=torch.float64, device="cuda")
        for t in range(9):
            u, v = t // 3, t % 3
            ref[:, :, u:u + 3, v:v + 3] += torch.einsum("oc,cixy->oixy", w2[:, :, u, v], w1)
    else:
        taps = layers[1].weight.double().reshape(c, 9) if kind == "block" else torch.ones(c, 1, dtype=torch.float64, device="cuda")
        ref = torch.einsum("oc,ct,ci->oit", w2[:, :, 0, 0], taps, w1[:, :, 0, 0]).reshape(wm.shape)
    assert ref.abs().max() < 2 ** 24
    wrong = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(60):
        wm.fill_(-0.5)
        dc.merge_chain(layers, [], wm, bm, None, dc.F32, ws)
        wrong += (wm.double() != ref).sum()
    assert int(wrong) == 0 and dc.async_status() == dc.OK


@pytest.mark.parametrize("n,h,w,ci,co,k,s", [(32, 28, 28, 32, 32, 5, 1), (3, 97, 97, 160, 72, 3, 2), (4, 61, 59, 64, 96, 3, 1), (128, 14, 14, 576, 96, 1, 1),
                                             (8, 14, 14, 384, 64, 3, 1), (2, 41, 43, 96, 112, 5, 2)])
def test_fp32_convs_by_bf16_terms_of_whole_numbers_are_exact_every_time(dc, n, h, w, ci, co, k, s):
    g = dc.geom(ci, co, 1, k, s, k // 2)
    assert dc.conv_kernel_name(n, h, w, g, dc.F32) == "k_conv_f32_tc"
    x, wf = (torch.from_numpy(whole_numbers(ci, d, 12)).cuda() for d in ((n, h, w, ci), (co, ci, k, k)))
    packed = torch.empty(dc.packed_bytes(g, dc.F32), dtype=torch.uint8, device="cuda")
    dc.pack_weights(wf, g, dc.F32, packed)
    ref = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), wf.double(), None, s, k // 2).permute(0, 2, 3, 1)
    ws, y = torch.zeros(dc.conv_workspace_bytes(), dtype=torch.uint8, device="cuda"), torch.empty(ref.shape, device="cuda")
    wrong = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(60):
        y.fill_(-0.5)
        dc.conv_forward(x, g, packed, None, dc.ACT_IDENTITY, None, y, ws)
        wrong += (y.double() != ref).sum()
    assert int(wrong) == 0 and dc.workspace_status(ws) == dc.OK


@pytest.mark.parametrize("algo", ["auto", "steps", "piece"])
@pytest.mark.parametrize("a,c,o", [(64, 4104, 64), (128, 4100, 130)])
def test_3x3_after_3x3_with_more_channels_between_than_the_tensor_core_takes(dc, algo, a, c, o):
    specs = [I.make_layer(89, 0, a, c, 3, 1, 1), I.make_layer(89, 1, c, o, 3, 1, 1)]
    if algo == "piece":                            # in the middle of a run, whose end reads what the composition wrote
        specs.append(I.make_layer(89, 2, o, 8, 1, 1, 0))
    W, b, k, s, p = O.merge_formula(specs, [])
    g, wm, bm, packed = run_merge(dc, specs, [], packed_dtype=dc.F32, algo=dc.MERGE_STEPS if algo == "steps" else dc.MERGE_AUTO)
    assert (g.k, g.stride, g.pad) == (k, s, p)
    assert O.rel_l2(wm.cpu().numpy(), W) <= TOL_W and O.rel_l2(bm.cpu().numpy(), b) <= TOL_W
    again = torch.full_like(packed, 7)
    dc.pack_weights(wm, g, dc.F32, again)
    assert torch.equal(packed, again)


def test_3x3_after_3x3_by_bf16_terms_of_what_is_not_finite(dc):
    """An infinity, a NaN and a value beyond the largest bf16 among the weights: infinities and NaN where 64 bits have them."""
    specs = [I.make_layer(88, 0, 104, 208, 3, 1, 1, with_bn=False), I.make_layer(88, 1, 208, 136, 3, 1, 1, with_bn=False)]
    w1, w2 = specs[0].weight, specs[1].weight
    w1[5, 7, 0, 1], w1[200, 103, 2, 2], w2[9, 11, 1, 1] = np.inf, np.nan, 3.4e38
    w1[11] *= 2.0 ** -20                           # the products of the largest value stay finite
    layers = [dc.DeviceLayer(s) for s in specs]
    g, ws_bytes = dc.merge_query(layers, [])
    wm, bm = torch.zeros(g.c_out, g.c_in, 5, 5, device="cuda"), torch.empty(g.c_out, device="cuda")
    dc.merge_chain(layers, [], wm, bm, None, dc.F32, torch.empty(ws_bytes, dtype=torch.uint8, device="cuda"))
    t1, t2 = (torch.from_numpy(w).double().cuda() for w in (w1, w2))
    ref = torch.zeros(136, 104, 5, 5, dtype=torch.float64, device="cuda")
    for u in range(3):
        for v in range(3):
            for p in range(3):
                for q in range(3):
                    ref[:, :, u + p, v + q] += (t2[:, :, u, v, None] * t1[None, :, :, p, q]).sum(1)
    wm = wm.double()
    assert torch.equal(torch.isnan(wm), torch.isnan(ref)) and torch.equal(torch.isinf(wm), torch.isinf(ref))
    fin = torch.isfinite(ref)
    big = ref.abs() > 1e20
    assert bool((wm[fin & big] / ref[fin & big] - 1).abs().max() < 1e-5) and int((fin & big).sum()) > 0
    assert ((wm - ref)[fin & ~big].norm() / ref[fin & ~big].norm()).item() <= 3e-7


@pytest.mark.parametrize("a,c,o,res,codes", [
    (160, 960, 160, [(0, 2)], "both"),         # two tiles of columns, twelve steps in eleven slots, the tile shared by five CTAs
    (96, 576, 96, [(0, 2)], "both"),           # shared by eight, the last with fewer steps
    (112, 672, 192, [], "both"),               # four sums of the products of the high terms
    (252, 700, 300, [], "f32"),                # the same; nothing a multiple of a tile or a step, slots used twice
    (36, 700, 250, [], "f32"),                 # columns and rows of the last tile that are not there
    (24, 1264, 40, [], "both"),                # packed orders that hold pixels, and taps, in their rows
    (40, 816, 24, [], "both"),
])
def test_blocks_by_bf16_terms_against_the_oracle(dc, a, c, o, res, codes):
    specs = [I.make_layer(90, 0, a, c, 1, 1, 0), I.make_layer(90, 1, c, c, 3, 1, 1, depthwise=True), I.make_layer(90, 2, c, o, 1, 1, 0)]
    _check_delivery(dc, specs, res, (dc.BF16, dc.F32) if codes == "both" else (dc.F32,))
    _check_delivery(dc, specs + [I.make_layer(90, 3, o, 16, 1, 1, 0)], res, (dc.F32,))         # as a piece
    assert dc.dwconv_status() == dc.OK


@pytest.mark.parametrize("a,c,o,res,codes", [
    (960, 320, 1280, [], "both"),              # a tile a CTA, twenty steps in ten slots
    (320, 1280, 320, [], "both"),              # shared by eight
    (332, 604, 333, [], "f32"),                # nothing a multiple of a tile or a step
    (72, 1500, 72, [], "both"),
    (504, 504, 504, [(0, 0)], "both"), (504, 504, 504, [(0, 0), (1, 1)], "both"), (504, 504, 504, [(0, 1)], "both"),
])
def test_1x1_pairs_by_bf16_terms_against_the_oracle(dc, a, c, o, res, codes):
    specs = [I.make_layer(91, 0, a, c, 1, 1, 0), I.make_layer(91, 1, c, o, 1, 1, 0)]
    _check_delivery(dc, specs, res, (dc.BF16, dc.F32) if codes == "both" else (dc.F32,))
    assert dc.dwconv_status() == dc.OK
    if not res:
        # sums of at most 128 products in the tensor core, then fp32 additions: 1.5e-7 measured at most; FMAs in runs of half or a quarter
        # of so many channels are 2.05e-7 or more away (so this also tells that they were not taken)
        _, wm, _, _ = run_merge(dc, specs, res, packed_dtype=dc.F32)
        assert O.rel_l2(wm.cpu().numpy(), O.merge_formula(specs, res)[0]) <= 1.9e-7


@pytest.mark.parametrize("block", [True, False])
def test_products_by_bf16_terms_of_what_is_not_finite(dc, block):
    """An infinity, a NaN and a value beyond the largest bf16 among the weights: infinities and NaN where 64 bits have them."""
    a, c, o = (96, 576, 96) if block else (320, 1280, 320)
    specs = [I.make_layer(92, 0, a, c, 1, 1, 0, with_bn=False), I.make_layer(92, 1, c, c, 3, 1, 1, depthwise=True, with_bn=False),
             I.make_layer(92, 2, c, o, 1, 1, 0, with_bn=False)]
    w1, wd, w2 = (s.weight for s in specs)
    w1[5, 7, 0, 0], w1[c - 1, a - 1, 0, 0], w2[9, 11, 0, 0] = np.inf, np.nan, 3.4e38
    w1[11] *= 2.0 ** -20                           # the products of the largest value stay finite
    specs = specs if block else specs[::2]
    layers = [dc.DeviceLayer(s) for s in specs]
    g, ws_bytes = dc.merge_query(layers, [])
    wm, bm = torch.zeros(g.c_out, g.c_in, g.k, g.k, device="cuda"), torch.empty(g.c_out, device="cuda")
    dc.merge_chain(layers, [], wm, bm, None, dc.F32, torch.empty(ws_bytes, dtype=torch.uint8, device="cuda"))
    t1, td, t2 = (torch.from_numpy(w).double().cuda() for w in (w1, wd, w2))
    taps = td[:, 0].reshape(c, 9) if block else torch.ones(c, 1, dtype=torch.float64, device="cuda")
    ref = torch.stack([((t2[:, :, 0, 0] * taps[:, t])[:, :, None] * t1[None, :, :, 0, 0]).sum(1) for t in range(taps.shape[1])], 2).reshape(wm.shape)
    wm = wm.double()
    assert torch.equal(torch.isnan(wm), torch.isnan(ref)) and torch.equal(torch.isinf(wm), torch.isinf(ref))
    fin = torch.isfinite(ref)
    big = ref.abs() > 1e20
    assert bool((wm[fin & big] / ref[fin & big] - 1).abs().max() < 1e-5) and int((fin & big).sum()) > 0
    assert ((wm - ref)[fin & ~big].norm() / ref[fin & ~big].norm()).item() <= 4e-7


@pytest.mark.parametrize("dw_first,a,o,res,codes", [
    (False, 160, 960, [], "both"),             # tiles of 64 input channels, the last one half filled
    (False, 72, 800, [], "both"),              # of 32
    (False, 150, 1000, [], "f32"),             # rows that are no whole 16-byte pieces
    (False, 24, 1600, [], "both"),             # a packed order that holds pixels in its rows
    (True, 1100, 180, [], "f32"),              # bias factors in two parts, tiles of 64
    (True, 1032, 48, [], "both"),              # the same, tiles of 16
    (True, 48, 24, [], "both"),                # taps in the rows
    (True, 400, 400, [(0, 0), (1, 1)], "both"), (False, 400, 400, [(0, 1)], "both"),
])
def test_1x1_and_depthwise_pairs_against_the_oracle(dc, dw_first, a, o, res, codes):
    mk = I.make_layer
    c = a if dw_first else o
    pair = [mk(93, 0, c, c, 3, 1, 1, depthwise=True), mk(93, 1, a, o, 1, 1, 0)]
    _check_delivery(dc, pair if dw_first else pair[::-1], res, (dc.BF16, dc.F32) if codes == "both" else (dc.F32,))


@pytest.mark.parametrize("before,a,c,s,res,codes", [
    ([], 96, 144, 2, [], "both"),
    ([], 24, 16, 1, [], "both"),               # packed orders that hold pixels in their rows
    ([], 48, 24, 1, [], "both"),               # and that do not
    ([], 50, 30, 1, [], "f32"), ([], 20, 12, 2, [], "f32"),        # rows that are no whole 16-byte pieces; tiles partly filled
    ([], 40, 40, 1, [(0, 0)], "both"), ([], 40, 40, 1, [(0, 0), (1, 1)], "both"), ([], 40, 40, 1, [(0, 1)], "both"),
    ([72, 24], 24, 144, 2, [], "both"),        # behind other layers
])
def test_3x3_then_depthwise_at_the_end_of_a_run(dc, before, a, c, s, res, codes):
    mk = I.make_layer
    chan = before + ([] if before and before[-1] == a else [a])
    specs = [mk(94, i, chan[i], chan[i + 1], 1, 1, 0) for i in range(len(chan) - 1)]
    specs += [mk(94, 7, a, c, 3, 1, 1), mk(94, 8, c, c, 3, s, 1, depthwise=True)]
    _check_delivery(dc, specs, res, (dc.BF16, dc.F32) if codes == "both" else (dc.F32,))
