"""Kernel variants and dispatch branches at the sizes where they can go wrong, against the CPU oracle.  Needs a B200."""
import numpy as np
import pytest
import torch

import lop_inputs as li
import paper_2507_05829_b200 as lop
from lop_inputs.workloads import NO_RESIDUAL, Segment, Workload, conv, pool
from oracle import chain as ochain
from paper_2507_05829_b200.chain import DeviceChain, to_host_f32
from test_gpu_parity import TOL, check_workload, one_layer, rel_err

pytestmark = pytest.mark.gpu


# ------------------------------------------------------------------------------------ CUDA-core convolution
SIMT_CASES = [  # k, s, p, d, cin, cout, N, H, W
    (3, 1, 1, 1, 16, 16, 1, 32, 32),       # small blocks, full
    (3, 2, 1, 1, 12, 21, 2, 17, 11),       # small blocks: ragged pixels and channels, K with a short last quad row
    (3, 1, 2, 2, 24, 40, 1, 70, 90),       # too many pixels for small blocks per SM, but Cin is no multiple of 16
    (1, 1, 0, 1, 16, 9, 1, 200, 161),      # few output channels: small blocks whatever the size
    (3, 1, 1, 1, 16, 64, 1, 150, 263),     # 128 x 64 tiles, ragged last tile
    (3, 1, 1, 1, 32, 100, 1, 93, 101),     # 64-wide tiles, ragged channels
    (1, 2, 0, 1, 48, 33, 2, 51, 77),       # odd channel count: scalar stores
    (5, 1, 2, 1, 80, 64, 1, 12, 14),       # K = 2000: operands do not fit the small block
    (7, 2, 3, 1, 3, 70, 1, 45, 52),        # thin input, K = 147 in three filter slices, ragged channels
    (1, 1, 0, 1, 1, 5, 1, 3, 3),           # the smallest
]


@pytest.mark.parametrize("case", SIMT_CASES)
def test_cuda_core_convolution_variants(case):
    k, s, p, d, cin, cout, N, H, W = case
    wl = one_layer(conv(cin, cout, k, s=s, p=p, d=d, act=li.ACT_SILU), N, H, W, dtype="f32")
    check_workload(wl, modes=("whole", "banded", "pipelined_copy"))


def test_cuda_core_convolution_takes_weights_of_any_alignment():
    """Weights four bytes off a vector boundary: the scalar kernel, the same bits."""
    wl = one_layer(conv(16, 24, 3, act=li.ACT_RELU), 1, 40, 33, dtype="f32")
    dc = DeviceChain(wl)
    x = dc.input_tensor()
    want = dc.run_whole(x).clone()
    l = wl.segments[0].layers[0]
    buf = torch.zeros(l.weight.size + 1, device="cuda")
    buf[1:] = torch.from_numpy(l.weight.reshape(-1)).cuda()
    sc, sh = torch.from_numpy(l.scale).cuda(), torch.from_numpy(l.shift).cuda()
    dc.plans[0].set_params(0, buf.data_ptr() + 4, sc.data_ptr(), sh.data_ptr())
    got = dc.run_whole(x)
    torch.cuda.synchronize()
    assert torch.equal(got, want)


# ------------------------------------------------------------------------------------ transfer of per-layer plans
@pytest.mark.parametrize("N,H,W,C,dtype,bands", [(1, 32, 32, 16, "f32", 4), (2, 7, 5, 3, "f32", 3), (3, 9, 13, 5, "bf16", 4), (1, 1, 1, 1, "f32", 1)])
def test_one_launch_brings_the_input_of_a_per_layer_plan(N, H, W, C, dtype, bands):
    """Rows of any length (no multiple of 16 bytes, images that start inside a vector), one band and all."""
    wl = one_layer(conv(C, 8, 1, p=0), N, H, W, dtype=dtype, n_bands=bands)
    dc = DeviceChain(wl, flags=lop.LOP_FLAG_REUSE_HALO | lop.LOP_FLAG_FORCE_SIMT)
    x = dc.pinned_input()
    dc.staging.fill_(float("nan"))
    dc.run_pipelined(x)
    torch.cuda.synchronize()
    assert dc.plans[0].last_copies() == 0 and dc.plans[0].last_launches() == 2
    assert torch.equal(dc.staging.cpu().view(-1), x.view(-1))
    assert rel_err(to_host_f32(dc.outs[-1]), ochain.run_workload(wl)) <= TOL[dtype]
    r = dc.plans[0].get_range(bands - 1, lop.LOP_INPUT)
    dc.staging.fill_(float("nan"))
    s = torch.cuda.current_stream().cuda_stream
    dc.plans[0].fetch_band(bands - 1, x.data_ptr(), dc.staging.data_ptr(), dc.ws[0].data_ptr(), s)
    torch.cuda.synchronize()
    assert torch.equal(dc.staging[:, r.new_lo:r.out_hi].cpu(), x[:, r.new_lo:r.out_hi])
    assert torch.isnan(dc.staging[:, :r.new_lo].float()).all() and torch.isnan(dc.staging[:, r.out_hi:].float()).all()


@pytest.mark.parametrize("dtype,C,N,H,W,bands,flags,copies", [
    ("f32", 8, 1, 512, 512, 5, lop.LOP_FLAG_REUSE_HALO, 2),                # the smallest input that comes in pieces
    ("f32", 8, 2, 519, 263, 7, 0, 2),                                      # odd sizes, bands that recompute their halo
    ("bf16", 12, 1, 611, 650, 3, lop.LOP_FLAG_FORCE_SIMT, 2),
    ("f32", 8, 1, 1024, 1024, 16, lop.LOP_FLAG_REUSE_HALO, 4),
])
def test_large_inputs_of_the_per_layer_kernels_come_in_pieces(dtype, C, N, H, W, bands, flags, copies):
    layers = [conv(C, C, 3, s=2, act=li.ACT_RELU), conv(C, C, 3, act=li.ACT_NONE), pool(C, 2, 2, 0)]
    layers[0].input_from, layers[1].input_from, layers[2].input_from = -1, 0, 1
    wl = Workload("pieces", dtype, N, H, W, C, [Segment(layers, bands)], seed=41)
    li.fill_parameters(wl)
    li.make_input(wl)
    check_workload(wl, flags=flags, modes=("banded", "pipelined"))
    dc = DeviceChain(wl, flags=flags)
    x = dc.pinned_input()
    for _ in range(3):                       # the staging tensor is written again only after the run before has read it
        dc.run_pipelined(x)
    torch.cuda.synchronize()
    assert dc.plans[0].last_copies() == copies
    assert torch.equal(dc.staging.cpu().view(-1), x.view(-1))


@pytest.mark.parametrize("dtype,C,H,W", [("f32", 16, 32, 32), ("f32", 8, 512, 512), ("bf16", 3, 60, 44)])
def test_streamed_runs_are_captured_in_a_graph(dtype, C, H, W):
    """One launch and one per layer, pieces on the side stream, the persistent kernel: replayed on another input."""
    wl = one_layer(conv(C, 16, 3, act=li.ACT_RELU), 1, H, W, dtype=dtype)
    dc = DeviceChain(wl, flags=lop.LOP_FLAG_REUSE_HALO)
    x = dc.pinned_input()
    dc.run_pipelined(x)                      # the first call makes streams, events and tables
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        dc.run_pipelined(x)
    other = torch.flip(x, [1]).clone()
    x.copy_(other)
    for _ in range(2):
        dc.outs[-1].zero_()
        graph.replay()
    torch.cuda.synchronize()
    dc.check_device()
    got = dc.outs[-1].clone()
    dc.run_banded(other.cuda())
    torch.cuda.synchronize()
    assert torch.equal(got, dc.outs[-1])


# ------------------------------------------------------------------------------------ operand ring and output units
RING_CASES = [  # k, s, p, cin, cout, N, H, W, residual
    (3, 1, 1, 64, 64, 1, 150, 143, True),      # kept weights: several tiles per CTA, one cut of the ring
    (1, 1, 0, 64, 256, 2, 90, 119, True),      # kept pointwise weights, two output units per tile
    (3, 1, 1, 128, 128, 1, 139, 141, False),   # 128-channel tiles: a filter row per weight box, a wait per row
    (5, 1, 2, 64, 128, 1, 17, 19, True),       # 40 KB weight boxes, two groups per chunk
    (3, 1, 1, 256, 80, 2, 9, 12, False),       # five output units of 16 channels: more than are in flight at a time
    (1, 1, 0, 192, 112, 3, 7, 5, True),        # seven units, tiles that fold images, rows beyond the band
    (3, 2, 1, 320, 48, 1, 21, 30, False),      # per-tap entries, the last one short
    (1, 1, 0, 16, 16, 1, 3, 3, True),          # the smallest tile
]


@pytest.mark.parametrize("case", RING_CASES)
def test_operand_ring_cuts_and_output_units(case):
    """One layer, then one with other tiles behind it (the ring is cut anew between them), bands and host output."""
    k, s, p, cin, cout, N, H, W, residual = case
    layers = [conv(cin, cout, k, s=s, p=p, act=li.ACT_RELU), conv(cout, cout, 1, p=0, act=li.ACT_NONE)]
    layers[0].input_from, layers[1].input_from = -1, 0
    if residual:
        layers[1].residual_from, layers[1].residual_pos = 0, li.RES_PRE_ACT
    wl = Workload("ring", "bf16", N, H, W, cin, [Segment(layers, 3)], seed=31)
    li.fill_parameters(wl)
    li.make_input(wl)
    want = check_workload(wl, flags=lop.LOP_FLAG_REUSE_HALO, modes=("whole", "banded", "pipelined"))["whole"][-1]
    dc = DeviceChain(wl, flags=lop.LOP_FLAG_REUSE_HALO)
    host = torch.zeros(dc.outs[-1].shape, dtype=dc.outs[-1].dtype).pin_memory()
    for _ in range(2):
        dc.run_pipelined(dc.pinned_input(), out_pinned=host)
        torch.cuda.synchronize()
        dc.check_device()
        assert np.array_equal(to_host_f32(host), want)


def _stack(layers, N, H, W, n_bands=3):
    for i, l in enumerate(layers):
        l.input_from = i - 1
    wl = Workload("stack", "bf16", N, H, W, layers[0].cin, [Segment(layers, n_bands)], seed=31)
    li.fill_parameters(wl)
    li.make_input(wl)
    return wl


@pytest.mark.parametrize("name", ["kept weights beside a wide image's gather scratch", "more boxes per chunk than entries"])
def test_operand_rings_with_little_room(name):
    """Rings that hold less than a full entry beside what is cut off them (tests/test_host_side.py walks them without a GPU)."""
    if name.startswith("kept"):
        wl = _stack([conv(3, 64, 7, s=2), conv(64, 32, 1), conv(32, 256, 3)], 1, 80, 1150)
    else:
        l = conv(512, 16, 1)
        l.kh, l.ph = 17, 8
        wl = _stack([l], 1, 26, 200)
    check_workload(wl, flags=lop.LOP_FLAG_REUSE_HALO, modes=("whole", "banded", "pipelined"))


def test_wide_resnet50_is_the_same_by_both_executors():
    """1152 columns: the gather's scratch takes 48 KB of the operand ring."""
    wl = li.build("resnet50", N=1, H=640, W=1152)
    outs = []
    for flags in (lop.LOP_FLAG_REUSE_HALO, lop.LOP_FLAG_REUSE_HALO | lop.LOP_FLAG_PER_LAYER):
        dc = DeviceChain(wl, flags=flags)
        dc.run_banded(dc.input_tensor())
        torch.cuda.synchronize()
        dc.check_device()
        outs.append(dc.outs[-1].clone())
        if not flags & lop.LOP_FLAG_PER_LAYER:
            dc.run_pipelined(dc.pinned_input())
            torch.cuda.synchronize()
            dc.check_device()
            assert torch.equal(dc.outs[-1], outs[0])
    assert torch.equal(outs[0], outs[1])


def test_units_that_workers_copy_out_are_taken_by_residual_loads():
    """Folded poolings and host output leave their units by the workers; residuals then arrive in the same units by bulk loads.
    Some seven tiles of each layer per CTA, four units."""
    layers = [conv(64, 64, 3, act=li.ACT_RELU), pool(64, 2, 2, 0), conv(64, 64, 1, act=li.ACT_RELU), conv(64, 64, 3, act=li.ACT_NONE)]
    wl = _stack(layers, 4, 368, 368, n_bands=8)
    layers[3].residual_from, layers[3].residual_pos = 1, li.RES_PRE_ACT
    ref = DeviceChain(wl, flags=lop.LOP_FLAG_REUSE_HALO | lop.LOP_FLAG_PER_LAYER)
    want = ref.run_banded(ref.input_tensor()).cpu()
    dc = DeviceChain(wl, flags=lop.LOP_FLAG_REUSE_HALO)
    x = dc.pinned_input()
    host = torch.zeros(dc.outs[-1].shape, dtype=dc.outs[-1].dtype).pin_memory()
    for _ in range(4):
        host.zero_()
        dc.run_pipelined(x, out_pinned=host)
        torch.cuda.synchronize()
        dc.check_device()
        assert torch.equal(host, want)


# ------------------------------------------------------------------------------------ gathered stems
STEM_CASES = [  # k, s, p, dilation, cin, cout, N, H, W
    (7, 2, 3, 1, 3, 64, 16, 150, 21),      # shared columns, four rows per gather item, a last item of three
    (7, 2, 3, 1, 3, 48, 5, 241, 33),       # two rows per item, rows whose bytes are no multiple of 16
    (3, 1, 1, 1, 3, 64, 1, 19, 1),         # one pixel wide
    (3, 1, 1, 1, 1, 16, 2, 9, 40),         # the shortest column: 3 of 8 values, runs of 24
    (3, 1, 1, 1, 8, 32, 1, 12, 17),        # 72 values in two chunks
    (5, 1, 4, 2, 3, 16, 1, 20, 23),        # dilated: patches
    (3, 2, 1, 1, 3, 32, 3, 33, 47),        # shared columns would be no smaller: patches
    (1, 2, 0, 1, 3, 16, 1, 11, 13),        # a pointwise stem
]


@pytest.mark.parametrize("case", STEM_CASES)
def test_gathered_stem_layouts(case):
    """Whole, band by band and streamed runs of the persistent kernel, and the per-layer kernels, on both layouts."""
    k, s, p, d, cin, cout, N, H, W = case
    layers = [conv(cin, cout, k, s=s, p=p, act=li.ACT_RELU)]
    layers[0].dh = layers[0].dw = d
    layers[0].input_from = -1
    wl = Workload("stem", "bf16", N, H, W, cin, [Segment(layers, 3)], seed=37)
    li.fill_parameters(wl)
    li.make_input(wl)
    check_workload(wl, flags=lop.LOP_FLAG_REUSE_HALO, modes=("whole", "banded", "pipelined"))
    check_workload(wl, flags=lop.LOP_FLAG_REUSE_HALO | lop.LOP_FLAG_PER_LAYER, modes=("whole", "banded"))


# ------------------------------------------------------------------------------------ 3x3 pooling, rows per item
POOL3_CASES = [  # s, p, C, N, H, W
    (2, 1, 8, 16, 151, 9),                 # four rows per item, the last item shorter
    (2, 0, 24, 9, 140, 21),                # two rows per item, no padding
    (1, 1, 64, 1, 12, 17),                 # one row per item, stride one
    (3, 1, 16, 16, 230, 7),                # four rows that share nothing
    (2, 1, 264, 1, 5, 3),                  # more channel vectors than a pass over the threads, columns next to both borders
]


@pytest.mark.parametrize("case", POOL3_CASES)
def test_pooling_rows_per_item(case):
    s, p, C, N, H, W = case
    wl = one_layer(pool(C, 3, s, p=p), N, H, W, n_bands=3)
    check_workload(wl, flags=lop.LOP_FLAG_REUSE_HALO, modes=("whole", "banded", "pipelined"))


# ------------------------------------------------------------------------------------ input fetched by the persistent kernel
@pytest.mark.parametrize("W", [1, 5, 8, 171, 777, 1000])
def test_fetched_rows_of_any_alignment(W):
    """Rows that start anywhere in a 128-byte line, shorter and longer than what a warp has in flight."""
    wl = one_layer(conv(3, 16, 3, act=li.ACT_RELU), 2, 11, W)
    check_workload(wl, flags=lop.LOP_FLAG_REUSE_HALO, modes=("pipelined",))


# ------------------------------------------------------------------------------------ GELU of the tensor-core epilogues
@pytest.mark.parametrize("flags", [0, lop.LOP_FLAG_PER_LAYER])
def test_gelu_over_its_whole_range(flags):
    """An identity layer: every output is the GELU of a bf16 value.  The epilogue's fp32 value is off by less than 1e-6 (its
    polynomial, and a handful of roundings near one), then it is rounded to bf16 once: half a unit in the last place."""
    from math import erfc
    C, x = 16, np.concatenate([np.linspace(-20.0, 20.0, 4001), np.logspace(-30, 30, 183), -np.logspace(-30, 30, 183), [0.0, -0.0, np.inf]])
    x = li.round_to_bf16(np.resize(x, 16 * 18 * C).astype(np.float32)).reshape(1, 16, 18, C)
    l = conv(C, C, 1, p=0, act=li.ACT_GELU)
    wl = one_layer(l, 1, 16, 18, dtype="bf16")
    l.weight = np.eye(C, dtype=np.float32).reshape(l.weight.shape)
    l.scale, l.shift = np.ones(C, np.float32), np.zeros(C, np.float32)
    # (0 times infinity is a NaN in the other channels of an infinite value's pixel)
    finite = np.isfinite(x).all(-1)
    got = to_host_f32((lambda dc: dc.run_whole(dc.input_tensor(x)))(DeviceChain(wl, flags=flags)))
    v = x.astype(np.float64)
    with np.errstate(invalid="ignore", over="ignore"):
        want = v * np.vectorize(lambda t: 0.5 * erfc(-t / np.sqrt(2.0)))(v)
    g, w = got[finite], want[finite]
    assert (np.abs(g - w) <= 2.0 ** -8 * np.abs(w) * (1 + 1e-3) + 1e-6 * np.minimum(np.abs(w), 1.0) + 1e-9).all()
    assert np.isposinf(got[np.isposinf(x)]).all()


@pytest.mark.parametrize("flags", [0, lop.LOP_FLAG_PER_LAYER])
def test_gelu_rounds_as_the_exact_function(flags):
    """Four million values of t in (-1, 0), where the result is small and its error shows: an fp32 value that is off by e is
    rounded to another bf16 than the exact one for a share of e over the spacing, which is 2^-8 to 2^-7 of the value, 0.0056 on
    the mean.  The bound is that of a mean error of one unit in fp32's last place, 6e-8 (measured: 7.9e-6; with a polynomial whose
    error was half as large again 1.4e-5)."""
    C, n = 64, 256
    rng = np.random.default_rng(11)
    x = li.round_to_bf16(rng.uniform(-0.9, -0.05, (1, n, n, C)).astype(np.float32))
    l = conv(C, C, 1, p=0, act=li.ACT_GELU)
    wl = one_layer(l, 1, n, n, dtype="bf16")
    w = np.eye(C) + 2.0 ** -9 * np.roll(np.eye(C), 1, axis=0)                  # two terms that the sum holds exactly: many values of t
    l.weight = w.astype(np.float32).reshape(l.weight.shape)
    l.scale, l.shift = rng.uniform(0.95, 1.05, C).astype(np.float32), rng.uniform(-0.04, 0.04, C).astype(np.float32)
    got = to_host_f32((lambda dc: dc.run_whole(dc.input_tensor(x)))(DeviceChain(wl, flags=flags)))
    t = torch.from_numpy(((x.astype(np.float64) @ w.T) * l.scale + l.shift).astype(np.float32)).double()    # (one rounding, as fmaf)
    want, e = np.frexp((0.5 * t * torch.erfc(-t / 2.0 ** 0.5)).numpy())
    want = np.ldexp(np.rint(want * 256.0) / 256.0, e)
    wrong = float((got != want).mean())
    assert (np.abs(got - want) <= 2.0 ** -7 * np.abs(want)).all()
    assert wrong < 6e-8 / 0.0056, wrong


# ------------------------------------------------------------------------------------ launches that begin before the previous one ended
@pytest.mark.parametrize("dtype,C,H,W,flags", [("bf16", 64, 40, 36, 0), ("bf16", 64, 40, 36, lop.LOP_FLAG_PER_LAYER), ("f32", 16, 32, 32, 0),
                                               ("f32", 64, 70, 61, 0), ("bf16", 5, 19, 23, lop.LOP_FLAG_FORCE_SIMT)])
def test_calls_in_a_row_wait_for_what_they_read(dtype, C, H, W, flags):
    """Two chains that read each other's output, called in turn with nothing between: the bits of calls with a
    synchronisation between them."""
    def chain(seed):
        wl = Workload("row", dtype, 1, H, W, C, [Segment([conv(C, C, 3, input_from=-1), pool(C, 3, 1, 1, input_from=0), conv(C, C, 1, p=0, input_from=1)], 2)], seed=seed)
        li.fill_parameters(wl)
        li.make_input(wl)
        return DeviceChain(wl, flags=flags)
    a, b = chain(5), chain(6)
    runs = []
    for between in (torch.cuda.synchronize, lambda: None):
        x = a.input_tensor()
        for call in range(6):
            x = (b if call % 2 else a).run_whole(x)
            between()
        torch.cuda.synchronize()
        runs.append((a.outs[-1].clone(), b.outs[-1].clone()))
    assert torch.isfinite(runs[0][1].float()).all() and runs[0][1].float().abs().max() > 0
    assert torch.equal(runs[0][0], runs[1][0]) and torch.equal(runs[0][1], runs[1][1])


@pytest.mark.parametrize("dtype,C,flags", [("f32", 16, 0), ("bf16", 64, 0), ("bf16", 64, lop.LOP_FLAG_PER_LAYER), ("bf16", 64, lop.LOP_FLAG_FORCE_SIMT)])
@pytest.mark.parametrize("streamed", [False, True])
def test_parameters_that_the_calls_before_have_written(dtype, C, flags, streamed):
    """A layer's filters are the output of the chain called before it, its scale and shift those of the one before that, other
    values in every turn: the bits of calls with a synchronisation between them.  (Streamed: a launch that brings the input
    stands between them.)"""
    side = {16: 12, 64: 24}[C]                                          # side x side x C values are C filters of 3x3xC
    makers = [one_layer(conv(C, C, 3, act=li.ACT_RELU), 1, side, side, dtype=dtype), one_layer(conv(16, C, 1, p=0), 1, 2, 1, dtype="f32"),
              one_layer(conv(C, C, 3, act=li.ACT_NONE), 1, 20, 18, dtype=dtype)]
    weights, affine, user = DeviceChain(makers[0], flags=flags), DeviceChain(makers[1]), DeviceChain(makers[2], flags=flags)
    per_channel = affine.outs[-1].data_ptr()
    user.plans[0].set_params(0, weights.outs[-1].data_ptr(), per_channel, per_channel + 4 * C)
    xs = [(weights.input_tensor() * f, affine.input_tensor() * f) for f in (1.0, -0.5, 0.25)]
    x, pinned = user.input_tensor(), user.pinned_input()
    runs = []
    for between in (torch.cuda.synchronize, lambda: None):
        got = []
        for turn in range(9):
            xw, xa = xs[turn % 3]
            for call in (lambda: affine.run_whole(xa), lambda: weights.run_whole(xw), lambda: user.run_pipelined(pinned) if streamed else user.run_whole(x)):
                out = call()
                between()
            got.append(out.clone())
        torch.cuda.synchronize()
        runs.append(got)
    assert all(torch.isfinite(t.float()).all() and t.float().abs().max() > 0 for t in runs[0])
    assert not torch.equal(runs[0][0], runs[0][1]) and torch.equal(runs[0][0], runs[0][3])
    assert all(torch.equal(a, b) for a, b in zip(*runs))


# ------------------------------------------------------------------------------------ K summed in parts by the CTAs of a cluster
SPLIT_CASES = [  # k, s, p, cin, cout, N, H, W, residual, activation; the parts that this layer and the 3x3 behind it are summed in
    (3, 1, 1, 512, 512, 1, 7, 7, li.RES_PRE_ACT, li.ACT_RELU, [4, 4]),          # one tile of pixels, every row of it in reach of padding
    (3, 1, 1, 256, 256, 3, 11, 16, li.RES_POST_ACT, li.ACT_SILU, [2, 2]),       # two chunks per part; ragged tiles
    (3, 1, 1, 256, 256, 1, 11, 16, li.RES_POST_ACT, li.ACT_SILU, [4, 4]),       # one chunk per part
    (3, 2, 1, 256, 512, 2, 15, 13, li.RES_NONE, li.ACT_RELU, [4, 4]),           # a box per tap, odd extents
    (1, 1, 0, 2048, 512, 8, 7, 7, li.RES_NONE, li.ACT_NONE, [4, 2]),            # pointwise
    (3, 1, 1, 256, 256, 8, 14, 14, li.RES_PRE_ACT, li.ACT_GELU, [2, 2]),
    (3, 2, 1, 128, 256, 1, 28, 26, li.RES_NONE, li.ACT_RELU, [2, 4]),           # two chunks: two parts at most
    (3, 1, 2, 128, 64, 1, 20, 18, li.RES_NONE, li.ACT_RELU, [1, 1]),            # too short a K: not split
]


def parts_of(dc):
    return [[plan.layer_parts(i) for i in range(plan.num_layers())] for plan in dc.plans]


@pytest.mark.parametrize("case", SPLIT_CASES)
def test_split_tiles(case):
    """Against the oracle, and bit for bit between the executors: a chain of two such layers (several split tiles per CTA,
    the second's partial sums behind the first's), one with a shortcut, in bands, streamed, into host memory."""
    k, s, p, cin, cout, N, H, W, res, act, parts = case
    l0 = conv(cin, cout, k, s=s, p=p, act=act, input_from=-1)
    layers = [l0, conv(cout, cout, 3, input_from=0, act=act, residual_from=0 if res != li.RES_NONE else NO_RESIDUAL, residual_pos=res)]
    wl = Workload("split", "bf16", N, H, W, cin, [Segment(layers, 3)], seed=31)
    li.fill_parameters(wl)
    li.make_input(wl)
    check_workload(wl, flags=lop.LOP_FLAG_REUSE_HALO, modes=("whole", "banded", "pipelined"))
    dc, per = DeviceChain(wl, flags=lop.LOP_FLAG_REUSE_HALO), DeviceChain(wl, flags=lop.LOP_FLAG_PER_LAYER)
    assert parts_of(dc) == parts_of(per) == [parts]
    want = per.run_whole(per.input_tensor())
    host = torch.empty(want.shape, dtype=want.dtype).pin_memory()
    for _ in range(3):                                                  # calls in a row, too
        got = dc.run_banded(dc.input_tensor())
        dc.run_pipelined(dc.pinned_input(), out_pinned=host)
    torch.cuda.synchronize()
    dc.check_device()
    assert torch.equal(got, want) and torch.equal(host, want.cpu())


MIXED_PARTS = [  # N, H, W, bands, segments of (k, s, cin, cout); the parts
    (3, 14, 14, 7, [[(3, 1, 512, 512), (3, 1, 512, 256), (3, 1, 256, 256), (3, 1, 256, 512), (3, 1, 512, 512), (3, 1, 512, 256)]], [[2, 4, 4, 2, 2, 4]]),
    (8, 7, 7, 3, [[(1, 1, 2048, 512), (3, 1, 512, 512), (1, 1, 512, 2048), (1, 1, 2048, 512), (3, 1, 512, 512)]], [[4, 2, 1, 4, 2]]),
    (3, 28, 31, 4, [[(3, 2, 128, 256), (3, 1, 256, 256), (3, 1, 256, 256)], [(3, 2, 256, 512), (3, 1, 512, 512)]], [[2, 2, 2], [4, 4]]),
]


@pytest.mark.parametrize("N,H,W,bands,segments,parts", MIXED_PARTS)
def test_tiles_of_two_parts_and_of_four_in_one_program(N, H, W, bands, segments, parts):
    """A CTA takes part in a tile of two parts and then in one of four, whose other CTAs need not have finished theirs: the bits
    of the per-layer kernels, in every one of many calls."""
    segs = [Segment([conv(cin, cout, k, s=s, p=k // 2, act=li.ACT_RELU, input_from=i - 1) for i, (k, s, cin, cout) in enumerate(ls)], bands) for ls in segments]
    wl = Workload("mixed", "bf16", N, H, W, segments[0][0][2], segs, seed=33)
    li.fill_parameters(wl)
    li.make_input(wl)
    dc, per = DeviceChain(wl, flags=lop.LOP_FLAG_REUSE_HALO), DeviceChain(wl, flags=lop.LOP_FLAG_PER_LAYER)
    assert parts_of(dc) == parts_of(per) == parts
    want = per.run_whole(per.input_tensor()).clone()
    assert torch.isfinite(want.float()).all() and want.float().abs().max() > 0
    x, pinned = dc.input_tensor(), dc.pinned_input()
    for _ in range(100):
        for call in (lambda: dc.run_banded(x), lambda: dc.run_pipelined(pinned)):
            dc.outs[-1].zero_()
            got = call()
            assert torch.equal(got, want)
    dc.check_device()


@pytest.mark.parametrize("case,pools", [(SPLIT_CASES[0], 0), (SPLIT_CASES[1], 0), (SPLIT_CASES[5], 0), (SPLIT_CASES[2], 3)])
def test_a_band_that_never_arrives_ends_a_launch_with_split_tiles(case, pools):
    """Band 1 is withheld (a dependency that the host never satisfies) with a limit of 4000 looks, one to two milliseconds: whoever
    waits for a part of a tile that will not come gives up with the rest, long before a wait of its own would run out (seconds);
    the status is reported once and the plan works again.  With poolings between, whose single rows are many items that the
    workers publish themselves, and the result stored to host memory, as split tiles are then, too: the workers may find their
    way to the publisher closed in front of a split tile."""
    k, s, p, cin, cout, N, H, W, res, act, parts = case
    layers = [conv(cin, cin, 1, p=0, input_from=-1)] + [pool(cin, 2, 1, 0, input_from=i) for i in range(pools)]
    layers += [conv(cin, cout, k, s=s, p=p, act=act, input_from=pools), conv(cout, cout, 3, act=act, input_from=pools + 1)]
    wl = Workload("withheld", "bf16", N, H, W, cin, [Segment(layers, 3)], seed=32)
    li.fill_parameters(wl)
    li.make_input(wl)
    dc = DeviceChain(wl, flags=lop.LOP_FLAG_REUSE_HALO | lop.LOP_FLAG_COPY_ENGINE)
    assert parts_of(dc)[0][-1] > 1
    plan, ws, x = dc.plans[0], dc.ws[0], dc.pinned_input()
    out = torch.empty_like(dc.outs[0], device="cpu").pin_memory() if pools else dc.outs[0]
    dc.run_pipelined(x, out_pinned=out if pools else None)
    torch.cuda.synchronize()
    good = out.clone()
    dc.check_device()
    for _ in range(2):
        plan.set_wait_limit(4000)
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        plan.run_pipelined_withheld(1, x.data_ptr(), dc.staging.data_ptr(), out.data_ptr(), ws.data_ptr(), torch.cuda.current_stream().cuda_stream)
        t1.record()
        torch.cuda.synchronize()
        assert t0.elapsed_time(t1) < 100.0
        with pytest.raises(lop.LopError) as e:
            plan.check_device(ws.data_ptr())
        assert e.value.status == -7
        plan.set_wait_limit(0)
        out.zero_()
        dc.run_pipelined(x, out_pinned=out if pools else None)
        torch.cuda.synchronize()
        dc.check_device()
        assert torch.equal(out, good)


def test_a_wait_limit_covers_as_much_time_as_it_says():
    """A band that never arrives with the largest limit that this call takes, 65536 looks of a quarter of a microsecond: 16.4 ms
    (a look takes a little longer than 256 ns where the clocks are lower, so there is no sharp bound from above)."""
    wl = li.build("vgg_block", H=44, W=36)
    dc = DeviceChain(wl, flags=lop.LOP_FLAG_REUSE_HALO | lop.LOP_FLAG_COPY_ENGINE)
    plan, ws, x = dc.plans[0], dc.ws[0], dc.pinned_input()
    dc.run_pipelined(x)
    torch.cuda.synchronize()
    plan.set_wait_limit(65536)
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record()
    plan.run_pipelined_withheld(1, x.data_ptr(), dc.staging.data_ptr(), dc.outs[0].data_ptr(), ws.data_ptr(), torch.cuda.current_stream().cuda_stream)
    t1.record()
    torch.cuda.synchronize()
    assert 15.5 < t0.elapsed_time(t1) < 100.0
    with pytest.raises(lop.LopError):
        plan.check_device(ws.data_ptr())


def test_a_late_band_is_waited_for_as_long_as_the_limit_says():
    """The bands' copies queue behind others that keep the link busy for 1.2 s, more than the roles behind the one that waits for
    rows used to wait (0.7 to 0.9 s); the limit is ten seconds."""
    wl = li.build("vgg_block", H=44, W=36)
    dc = DeviceChain(wl, flags=lop.LOP_FLAG_REUSE_HALO | lop.LOP_FLAG_COPY_ENGINE)
    x = dc.pinned_input()
    good = dc.run_pipelined(x).clone()
    big = torch.empty(128 << 20, dtype=torch.uint8).pin_memory()
    there, side = torch.empty_like(big, device="cuda"), torch.cuda.Stream()
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)

    def copies(n):
        for _ in range(n):
            there.copy_(big, non_blocking=True)
    with torch.cuda.stream(side):
        copies(2)
        t0.record()
        copies(8)
        t1.record()
    torch.cuda.synchronize()
    dc.outs[-1].zero_()
    dc.plans[0].set_wait_limit(1 << 25)
    with torch.cuda.stream(side):
        copies(int(1200.0 * 8 / t0.elapsed_time(t1)))
    dc.run_pipelined(x)
    torch.cuda.synchronize()
    dc.check_device()
    assert torch.equal(dc.outs[-1], good)
