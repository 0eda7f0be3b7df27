"""The library's host side -- planner, executors, program builder -- compiled against stand-ins for the CUDA runtime and the
kernel launches (tests/host_side/runtime.cpp): what it would launch is checked without launching anything."""
import ctypes
import os
import random
import subprocess
from types import SimpleNamespace

import pytest

import lop_inputs as li
import paper_2507_05829_b200 as lop
from lop_inputs.workloads import Segment, Workload, conv, pool
from paper_2507_05829_b200 import binding
from paper_2507_05829_b200.chain import _FIELDS

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DEVICE = 1 << 46                             # where the stand-in runtime's device addresses begin
HOST = 0x10000000                            # a host buffer


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    csrc = os.path.join(ROOT, "paper_2507_05829_b200", "csrc")
    out = str(tmp_path_factory.mktemp("host_side") / "host_side.so")
    subprocess.check_call(["/usr/local/cuda/bin/nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O1", "-cudart", "none",
                           "-Xcompiler", "-fPIC", "-Xlinker", "-Bsymbolic", "-shared", "-I", os.path.join(ROOT, "include"), "-I", csrc, "-o", out] +
                          [os.path.join(csrc, f) for f in ("lop_plan.cpp", "lop_program.cu", "lop_exec.cu")] +
                          [os.path.join(ROOT, "tests", "host_side", "runtime.cpp")])
    return out


@pytest.fixture
def host(library, monkeypatch):
    """The binding on top of the stand-in build, for one test."""
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "LIB_PATH", library)
    monkeypatch.setattr(binding._build, "needs_build", lambda: False)
    L = binding.lib()
    L.host_side_log.restype = ctypes.c_char_p
    L.host_side_pin.argtypes = [ctypes.c_size_t, ctypes.c_size_t]
    L.host_side_pin(HOST, 1 << 30)
    chains = []

    def chain(wl, flags=lop.LOP_FLAG_REUSE_HALO):
        chains.append(Chain(wl, flags))
        return chains[-1]

    yield SimpleNamespace(lib=L, chain=chain)
    for c in chains:                          # (a plan must not outlive the library that made it)
        for p in c.plans:
            p.destroy()


class Chain:
    """The plans of a workload with made-up device addresses."""

    def __init__(self, wl, flags):
        self.plans, (H, W, C) = [], (wl.H, wl.W, wl.C)
        for seg in wl.segments:
            layers = [SimpleNamespace(weight_ptr=DEVICE + 4096, scale_ptr=DEVICE, shift_ptr=DEVICE, **{f: getattr(l, f) for f in _FIELDS})
                      for l in seg.layers]
            self.plans.append(binding.Plan(layers, wl.N, H, W, C, lop.LOP_BF16 if wl.dtype == "bf16" else lop.LOP_F32, seg.n_bands, flags))
            H, W, C = self.plans[-1].out_shape(len(layers) - 1)
        self.ws = [DEVICE + (1 << 44) + (i << 36) for i in range(len(self.plans))]
        self.outs = [DEVICE + (2 << 44) + (i << 36) for i in range(len(self.plans))]
        self.staging = DEVICE + (3 << 44)

    def banded(self):
        binding.run_chain_banded(self.plans, self.staging, self.outs, self.ws, None)

    def pipelined(self, host_out=None):
        outs = self.outs[:-1] + [host_out or self.outs[-1]]
        if len(self.plans) == 1:
            return self.plans[0].run_pipelined(HOST, self.staging, outs[0], self.ws[0], None)
        binding.run_chain_pipelined(self.plans, HOST, self.staging, outs, self.ws, None)


# ------------------------------------------------------------------------------------ operand rings
def check_rings(host, wl):
    c = host.chain(wl)
    for run in (c.banded, c.pipelined, lambda: c.pipelined(host_out=HOST + (1 << 29))):
        run()
        assert host.lib.host_side_walk_rings() == 0, (wl.name, wl.H, wl.W)


@pytest.mark.parametrize("W", [1024, 1088, 1104, 1120, 1136, 1152, 1168, 1200])
@pytest.mark.parametrize("H", [256, 640, 1152])
def test_every_ring_entry_fits_its_ring_in_wide_resnets(host, H, W):
    """A wide image leaves the operand ring little room: the gather's scratch holds its rows."""
    check_rings(host, li.build("resnet50", with_data=False, N=1, H=H, W=W))


def test_every_ring_entry_fits_its_ring_behind_a_stem(host):
    rnd = random.Random(11)
    for i in range(60):
        c = rnd.choice([32, 64])
        layers = [conv(3, c, rnd.choice([3, 7]), s=rnd.choice([1, 2]))]
        for _ in range(rnd.randint(1, 4)):
            cout = rnd.choice([16, 32, 48, 64, 80, 128, 256, 512])
            layers.append(conv(c, cout, rnd.choice([1, 1, 3, 3, 5]), s=rnd.choice([1, 1, 1, 2])))
            c = cout
        for j, l in enumerate(layers):
            l.input_from = j - 1
        check_rings(host, Workload("stack %d" % i, "bf16", 1, rnd.randint(64, 640), rnd.randint(600, 1250), 3, [Segment(layers, 4)]))


@pytest.mark.parametrize("cout,W", [(256, 512), (512, 900), (256, 1150)])
def test_every_ring_entry_fits_its_ring_with_many_kept_weights(host, cout, W):
    """72 KB of kept weights beside the gather's scratch."""
    layers = [conv(3, 64, 7, s=2), conv(64, 32, 1), conv(32, cout, 3)]
    for j, l in enumerate(layers):
        l.input_from = j - 1
    check_rings(host, Workload("kept", "bf16", 1, 900, W, 3, [Segment(layers, 4)]))


def test_a_group_of_boxes_fits_the_rings_entries(host):
    """Seventeen boxes of one filter column each per chunk, with room for all of them: more than a ring has entries."""
    l = conv(512, 16, 1)
    l.kh, l.ph, l.input_from = 17, 8, -1
    wl = Workload("column", "bf16", 1, 26, 200, 512, [Segment([l], 2), Segment([conv(16, 16, 1, input_from=-1)], 1)])
    check_rings(host, wl)


def commands(host, run):
    """The stream commands and launches of one call, as (command, stream, ...) tuples."""
    host.lib.host_side_clear()
    run()
    return [tuple(line.split()) for line in host.lib.host_side_log().decode().splitlines()]


@pytest.mark.parametrize("layer", [li.dwconv(64, 7), li.layernorm(64), pool(64, 3, 2, 1), conv(64, 64, 1)])
def test_a_program_without_a_convolution_leaves_shared_memory_to_l1(host, layer):
    layer.input_from = -1
    c = host.chain(Workload("one", "bf16", 2, 56, 56, 64, [Segment([layer], 4)]))
    for run in (c.banded, c.pipelined):
        smem = [int(x[2]) for x in commands(host, run) if x[0] == "persistent"]
        assert len(smem) == 1 and (smem[0] > 200 * 1024) == (layer.op == conv(1, 1, 1).op) and smem[0] <= 227 * 1024
        assert layer.op == conv(1, 1, 1).op or smem[0] <= (1 + 4 + 4 + 64) * 1024          # alignment, tables, units, scratch


# ------------------------------------------------------------------------------------ the streamed input's transport


@pytest.mark.parametrize("name", ["single_conv", "vgg_block", "resnet18"])
def test_an_address_that_is_no_longer_page_locked_is_copied_from(host, name):
    """The same address, page-locked, then an ordinary allocation's, then page-locked again: fp32, bf16, a chain of plans."""
    c = host.chain(li.build(name, with_data=False))
    for pinned in (True, False, True):
        host.lib.host_side_pin(HOST, (1 << 30) if pinned else 0)
        copies = [x for x in commands(host, c.pipelined) if x[0] == "copy"]
        assert bool(copies) == (not pinned), (name, pinned)


@pytest.mark.parametrize("flags", [0, lop.LOP_FLAG_REUSE_HALO])
@pytest.mark.parametrize("N,H,bands,pieces", [(1, 511, 8, 1), (1, 512, 8, 2), (2, 517, 3, 2), (1, 2047, 5, 2), (1, 2048, 32, 4), (3, 2048, 2, 2),
                                              (1, 4096, 1, 1), (1, 2050, 4000, 4)])
def test_a_large_input_of_the_per_layer_kernels_arrives_while_it_is_computed(host, N, H, bands, pieces, flags):
    """From 8 MB on, a 512-column fp32 input of 8 channels comes in pieces, and each layer's rows are computed once, as
    far as the rows that have arrived allow."""
    layers = [conv(8, 8, 5, s=2), conv(8, 8, 3)]
    layers[0].input_from, layers[1].input_from = -1, 0
    c = host.chain(Workload("two", "f32", N, H, 512, 8, [Segment(layers, bands)]), flags=flags)
    plan, log = c.plans[0], commands(host, c.pipelined)
    side = {x[1] for x in log if x[0] == "copy"}
    copies = [int(x[2]) for x in log if x[0] == "copy"]
    convs = [(int(x[3]), int(x[4])) for x in log if x[0] == "conv"]
    fetches = [x for x in log if x[0] == "fetch"]
    assert (len(copies), len(fetches)) == ((0, 1) if pieces == 1 else (pieces, 0))
    assert sum(copies) == (N * H * 512 * 32 if copies else 0) and side.isdisjoint({"0"}) and len(convs) == 2 * pieces
    assert (plan.last_copies(), plan.last_launches()) == (len(copies), len(convs) + len(fetches))
    for layer in range(2):
        rows = convs[layer::2]
        assert rows[0][0] == 0 and rows[-1][1] == plan.out_shape(layer)[0]
        assert all(a[1] == b[0] for a, b in zip(rows, rows[1:]))
    # a piece's layers follow the wait for its copy, and need no row that comes later
    arrived, row, waited, recorded = {}, 0, 0, [x[2] for x in log if x[0] == "record" and x[1] in side]
    for e, n in zip(recorded, copies):
        row += n // (N * 512 * 32)
        arrived[e] = row
    for x in log:
        if x[0] == "wait" and x[1] == "0":
            waited = arrived[x[2]]
        elif x[0] == "conv" and copies and int(x[4]) == convs[2 * list(arrived.values()).index(waited)][1]:
            assert min(H, (int(x[4]) - 1) * 2 - 2 + 5) <= waited
