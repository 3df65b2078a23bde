"""Host paths of the library without a GPU, on a stand-in for the CUDA runtime (_fake_cuda.py): the
launches that a call makes, their arguments, and what it copies, waits for and gives back."""
import ctypes
import shutil

import pytest

import _fake_cuda as F

LB_OK, LB_ENOMEM, LB_ECUDA, LB_ESTATE = 0, -2, -3, -7
P = ctypes.c_void_p
I32, I64 = ctypes.c_int32, ctypes.c_int64


@pytest.fixture(scope="module")
def built(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    return F.build(tmp_path_factory.mktemp("fake"))


@pytest.fixture
def fake(built):
    built.reset()
    yield built
    built.reset()


class ConvArgs(ctypes.Structure):            # csrc/lb_conv.h
    _fields_ = [("x", P), ("ldx", I64), ("xoff", I32), ("w", P), ("wp", P), ("bias", P), ("y", P), ("yf", P),
                ("ldy", I64), ("yoff", I32), ("B", I32), ("H", I32), ("W", I32), ("Ci", I32), ("Co", I32), ("act", I32),
                ("ym", P), ("ldm", I64), ("moff", I32), ("up", P), ("ldu", I64), ("yf2", P), ("w_late", I32)]


class PackLayer(ctypes.Structure):
    _fields_ = [("w", P), ("Ci", I32), ("Co", I32), ("fwd", P), ("dgrad", P), ("wt", P)]


def arguments(fake, kernel, struct):
    """The first argument of every launch of `kernel` from here on, as copies."""
    seen = []

    def f(name, args):
        if kernel in name.decode():
            seen.append(struct.from_buffer_copy(ctypes.cast(args[0], ctypes.POINTER(struct)).contents))
    fake.hook(f)
    return seen


def both(fake, *pairs):
    seen = [[] for _ in pairs]

    def f(name, args):
        for k, (kernel, struct) in enumerate(pairs):
            if kernel in name.decode():
                seen[k].append(struct.from_buffer_copy(ctypes.cast(args[0], ctypes.POINTER(struct)).contents))
    fake.hook(f)
    return seen


# ---- single convolution layers

GZ, GX, WT, X, GW, GB = (k << 40 for k in range(1, 7))      # addresses that nothing touches


@pytest.fixture
def conv(fake):
    for a in (GZ, GX, WT, X, GW, GB):
        fake.memory(a, 1 << 39)
    fake.L.lb_conv3x3_dgrad.argtypes = [P, P, P, I32, I32, I32, I32, I32, P]
    fake.L.lb_conv3x3_wgrad.argtypes = [P, P, P, P, I32, I32, I32, I32, I32, P]
    fake.L.lb_conv3x3.argtypes = [P, I64, I32, P, P, P, P, I64, I32, I32, I32, I32, I32, I32, I32, P]
    yield fake
    for a in (GZ, GX, WT, X, GW, GB):
        fake.memory(a, 0)


@pytest.mark.parametrize("B,H,W,tc", [(1, 32768, 65535, True), (1, 32768, 65536, False), (2, 32768, 32768, False),
                                      (3, 32768, 32768, False), (1, 64, 64, True)])
def test_data_gradient_reads_the_weights_in_the_form_that_its_kernel_takes(conv, B, H, W, tc):
    # from 2^31 pixels on the mma.sync kernel runs (the tcgen05 one has 32-bit pixel indices): it reads
    # w' as [9][Ci][Co], the other one the packed form
    packs, args = both(conv, ("k_conv_pack", PackLayer), ("k_conv3x3" if not tc else "k_conv_tc", ConvArgs))
    assert conv.L.lb_conv3x3_dgrad(GZ, WT, GX, B, H, W, 16, 32, None) == LB_OK
    assert len(packs) == 1 and len(args) == 1
    if tc:
        assert args[0].wp and args[0].wp == packs[0].dgrad
    else:
        assert args[0].w and args[0].w == packs[0].wt
    assert (args[0].x, args[0].y, args[0].Ci, args[0].Co) == (GZ, GX, 32, 16)


# ---- the network's output

@pytest.mark.parametrize("kind,device,shift,room,direct", [
    (F.DEVICE, 0, 0, 0, True), (F.DEVICE, 0, 4, 0, True), (F.DEVICE, 0, 1, 0, False), (F.DEVICE, 0, 2, 0, False),
    (F.DEVICE, 1, 0, 0, False), (F.HOST, 0, 0, 0, False), (F.MANAGED, 0, 0, 0, False), (0, -2, 0, 0, False),
    (F.DEVICE, 0, 0, -4, False)])
def test_network_output_goes_by_copy_where_a_kernel_must_not_write(fake, kind, device, shift, room, direct):
    # memory of this device at a multiple of four bytes: the head convolution stores there; host, managed
    # or another device's memory, an odd address, an end outside: the runtime's copy, which handles or refuses it
    L = fake.L
    L.lb_net_create.argtypes = [I32, I32, I32, ctypes.c_uint64, P, P]
    L.lb_net_forward.argtypes = [P, P, P]
    L.lb_net_output.argtypes, L.lb_net_output.restype = [P], P
    L.lb_net_destroy.argtypes = [P]
    n = P()
    assert L.lb_net_create(1, 8, 16, 1, None, ctypes.byref(n)) == LB_OK
    nbytes = 4 * 8 * 16 * 16
    base = 7 << 40
    if kind:
        fake.memory(base, nbytes + shift + room, kind, device)
    y = base + shift
    x = ctypes.create_string_buffer(2 * 8 * 16 * 16)
    if not kind:                                 # a plain host buffer
        buf = ctypes.create_string_buffer(nbytes)
        y = ctypes.addressof(buf)
    fake.clear()
    seen = arguments(fake, "k_conv_tc", ConvArgs)
    assert L.lb_net_forward(n, x, y) == LB_OK
    assert [a.yf2 for a in seen if a.yf2] == ([y] if direct else [])
    copies = [c for c in fake.calls("cudaMemcpyAsync") if int(c[1], 16) == y]
    assert [(int(c[2], 16), int(c[3])) for c in copies] == ([] if direct else [(L.lb_net_output(n), nbytes)])
    fake.hook(None)
    L.lb_net_destroy(n)
    fake.memory(base, 0)


# ---- lattices

def solver(fake, nx, ny, rings=0, every=4, stream=None, **kw):
    """A handle on the stand-in, with `rings` small rings, ready to step."""
    from paper_2209_14889_gb300 import lb
    L = fake.L
    base = dict(nx=nx, ny=ny, tau=0.8, rho0=1.0, K1111=2e-3, K1122=1e-3, K2222=1e-3, K1212=1e-3, eta_p=0.1,
                lambda_steps=0.0, Dp=0.05, alpha=-0.9, beta=1.0, xi=1.1, Gamma=1.0, kappa=1e-3, P_cap=0.99,
                director_angle=0.0, ericksen=1, precision=0, readout_every=every, max_samples=16)
    base.update(kw)
    h = P()
    assert L.lb_create(ctypes.byref(lb.lb_params(**base)), P(stream), ctypes.byref(h)) == LB_OK
    if rings:
        import math
        rd = (lb.lb_ring * rings)(*[lb.lb_ring(n_nodes=12, k_spring=0.1, eps_angle=0.01, l_eq=1.0) for _ in range(rings)])
        X = [c for r in range(rings) for k in range(12)
             for c in (nx / 2 + 0.1 * r + 2 * math.cos(k * math.pi / 6), ny / 2 + 2 * math.sin(k * math.pi / 6))]
        X = (ctypes.c_double * len(X))(*X)
        L.lb_set_body.argtypes = [P, I32, P, P]
        assert L.lb_set_body(h, rings, rd, X) == LB_OK
    L.lb_init_fields.argtypes = [P, P]
    assert L.lb_init_fields(h, None) == LB_OK
    L.lb_step.argtypes = [P, I64]
    L.lb_set_kernel.argtypes = [P, I32]
    L.lb_destroy.argtypes = [P]
    return h


def test_strip_step_behind_a_launch_with_the_node_tail_starts_when_that_has_ended(fake):
    # it reads the state by the read-only path, which the launch before must no longer write
    from paper_2209_14889_gb300 import lb
    h = solver(fake, 128, 64, rings=1)
    assert fake.L.lb_step(h, 2) == LB_OK
    assert fake.L.lb_set_kernel(h, lb.LB_KERNEL_STRIP) == LB_OK
    fake.clear()
    assert fake.L.lb_step(h, 3) == LB_OK
    assert [c[-1] for c in fake.launches("k_strip")] == ["0", "1", "1"]
    fake.L.lb_destroy(h)


def gradient_calls(L):
    return {"dgrad": lambda s: L.lb_conv3x3_dgrad(GZ, WT, GX, 1, 9, 40, 32, 16, s),
            "wgrad": lambda s: L.lb_conv3x3_wgrad(X, GZ, GW, GB, 1, 9, 40, 32, 16, s)}


@pytest.mark.parametrize("which", ["dgrad", "wgrad"])
@pytest.mark.parametrize("kernel", [0, 1])
def test_single_layer_gradients_return_when_they_are_done(conv, which, kernel):
    # the results may be read from any stream or freed; a fault of their kernels is their own return code
    s = 0x77770
    conv.L.lb_conv_kernel(kernel)
    call = gradient_calls(conv.L)[which]
    assert call(s) == LB_OK
    kinds = [c[0] for c in conv.calls()]
    last = len(kinds) - 1 - kinds[::-1].index("launch")
    assert ["cudaStreamSynchronize", hex(s)] in conv.calls()[last:]
    live = conv.L.fake_live()
    conv.fail("cudaStreamSynchronize", 1, 700)
    assert call(s) == LB_ECUDA
    assert conv.L.fake_live() == live
    conv.L.lb_conv_kernel(1)


# ---- batches

def batch(fake, handles):
    L = fake.L
    for f, a in (("lb_batch_create", [P, I32, P]), ("lb_batch_step", [P, I64]), ("lb_batch_set_shape", [P, I32, I32]),
                 ("lb_batch_set_persistent", [P, I32]), ("lb_batch_destroy", [P]), ("lb_batch_uses_graph", [P])):
        getattr(L, f).argtypes = a
    arr = (P * len(handles))(*[h.value for h in handles])
    b = P()
    assert L.lb_batch_create(arr, len(handles), ctypes.byref(b)) == LB_OK
    return b


SIZES = [dict(nx=128, ny=96, rings=1), dict(nx=64, ny=64), dict(nx=160, ny=80, rings=1, Dp=0.3, diffusion_substeps=3),
         dict(nx=71, ny=53)]


@pytest.mark.parametrize("call", ["cudaMalloc", "cudaMemcpy", "cudaStreamCreateWithPriority", "cudaEventCreateWithFlags"])
@pytest.mark.parametrize("nth", [1, 2, 3])
@pytest.mark.parametrize("change", ["shape", "persistent"])
def test_batch_with_a_plan_that_failed_launches_nothing(fake, call, nth, change):
    # a change of plan that the runtime refuses half way: the launches and the graph of the former plan
    # read tables that are gone or half replaced
    L = fake.L
    hs = [solver(fake, **kw) for kw in SIZES]
    b = batch(fake, hs)
    if change == "persistent":
        assert L.lb_batch_set_persistent(b, 1) == LB_OK
    assert L.lb_batch_step(b, 8) == LB_OK
    change = (lambda: L.lb_batch_set_shape(b, -1, 1)) if change == "shape" else (lambda: L.lb_batch_set_persistent(b, 0))
    fake.fail(call, nth)
    rc = change()
    fake.fail("")
    fake.clear()
    again = L.lb_batch_step(b, 4)
    if rc != LB_OK:
        assert again == LB_ESTATE
        assert not fake.calls("launch") and not fake.calls("cudaGraphLaunch")
        assert change() == LB_OK and L.lb_batch_step(b, 4) == LB_OK
    else:
        assert again == LB_OK
    L.lb_batch_destroy(b)
    for h in hs:
        L.lb_destroy(h)


def test_batch_of_one_group_makes_no_streams_it_does_not_use(fake):
    # creating a batch: one buffer for the plan, streams and events of the groups that fork only
    hs = [solver(fake, 128, 96, rings=1)]
    fake.clear()
    b = batch(fake, hs)
    assert len(fake.calls("cudaMalloc")) <= 5 and not fake.calls("cudaStreamCreateWithPriority")
    assert fake.L.lb_batch_step(b, 9) == LB_OK
    fake.L.lb_batch_destroy(b)
    fake.L.lb_destroy(hs[0])


@pytest.mark.parametrize("shapes", [(0, 0, 0, 0), (4, 1, 0, 3), (2, 2, 2, 2)])
@pytest.mark.parametrize("members", [(0,), (2,), (0, 1), (0, 1, 2, 3)])
def test_batch_launches_wait_for_each_other_through_streams_and_events_that_exist(fake, shapes, members):
    # every launch of the steps is on a stream that was created, every event waited for was recorded before
    L = fake.L
    hs = [solver(fake, **SIZES[i]) for i in members]
    fake.clear()
    b = batch(fake, hs)
    for k, i in enumerate(members):
        if shapes[i] != 4 or i == 0:
            assert L.lb_batch_set_shape(b, k, shapes[i]) == LB_OK
    made = {c[1] for c in fake.calls() if c[0].startswith(("cudaStreamCreate", "cudaEventCreate"))}
    fake.clear()
    assert L.lb_batch_step(b, 9) == LB_OK
    recorded = set()
    for c in fake.calls():
        if c[0] == "cudaEventRecord":
            recorded.add(c[1])
            assert c[1] in made
        elif c[0] == "cudaStreamWaitEvent":
            assert c[2] in recorded
        elif c[0] == "launch":
            assert c[7] in made
    L.lb_batch_destroy(b)
    for h in hs:
        L.lb_destroy(h)


@pytest.mark.parametrize("nx,ny,scalar,rings,grid", [
    (96, 96, 0, 0, (12, 12)), (224, 224, 0, 0, (14, 28)), (250, 250, 0, 0, (8, 16)), (320, 320, 0, 0, (20, 20)),
    (384, 384, 0, 0, (12, 24)), (384, 384, 1, 0, (12, 24)), (512, 512, 1, 0, (16, 32)), (64, 1024, 0, 0, (2, 64)),
    (250, 250, 0, 1, (16, 32)), (384, 384, 0, 1, (24, 24)), (512, 512, 1, 1, (32, 64))])
def test_tile_shape_by_size_and_rings(fake, nx, ny, scalar, rings, grid):
    # the grid of the step's launch: 8x8, 16x8, 16x16 or 32x16 cells per CTA; a lattice without rings leaves the
    # small tiles sooner
    from paper_2209_14889_gb300 import workloads as W
    kw = dict(model=1, ericksen=0, K1111=1.875e-3, K1122=0.0, K2222=1.875e-3, K1212=0.9375e-3) if scalar else {}
    h = solver(fake, nx, ny, rings=rings, **kw)
    fake.clear()
    assert fake.L.lb_step(h, 1) == LB_OK
    assert [(int(c[2]), int(c[3])) for c in fake.launches("k_fused")] == [grid]
    fake.L.lb_destroy(h)


@pytest.mark.parametrize("B,H,W,Ci,Co,minb", [(1, 32, 32, 1024, 256, 4), (2, 64, 64, 512, 512, 4), (1, 1024, 1024, 16, 16, 5),
                                              (16, 64, 64, 128, 128, 4), (1, 2048, 2048, 16, 32, 5)])
def test_mma_convolution_takes_registers_or_occupancy_by_its_waves(conv, B, H, W, Ci, Co, minb):
    conv.L.lb_conv_kernel(0)
    assert conv.L.lb_conv3x3(X, Ci, 0, WT, None, GX, None, Co, 0, B, H, W, Ci, Co, 1, None) == LB_OK
    conv.L.lb_conv_kernel(1)
    assert ["k_conv3x3ILi%dE" % minb in c[1] for c in conv.launches("k_conv3x3")] == [True]


@pytest.mark.parametrize("ldy,shift,odd", [(16, 0, False), (16, 2, True), (17, 0, True), (18, 4, False), (17, 2, True)])
def test_mma_convolution_stores_pairs_at_even_addresses_only(conv, ldy, shift, odd):
    conv.L.lb_conv_kernel(0)
    assert conv.L.lb_conv3x3(X, 16, 0, WT, None, GX + shift, None, ldy, 0, 1, 9, 9, 16, 16, 1, None) == LB_OK
    conv.L.lb_conv_kernel(1)
    assert [c[1].split("k_conv3x3IL")[1].split("EE")[0].endswith("b1") for c in conv.launches("k_conv3x3")] == [odd]


def test_work_is_split_over_the_sms_of_the_current_device(conv):
    # device 0 of the stand-in has 152 SMs, device 1 has 76
    def grid(dev):
        conv.L.fake_device(dev)
        conv.clear()
        assert conv.L.lb_conv3x3_wgrad(X, GZ, GW, GB, 4, 256, 256, 32, 32, None) == LB_OK
        return conv.launches("k_wgrad_tc")[0][2]
    assert [grid(d) for d in (0, 1, 0)] == ["152", "76", "152"]


@pytest.mark.parametrize("H,W,mt", [(1, 100000, 1), (4, 100000, 1), (8, 100000, 2), (9, 100000, 4), (1024, 1024, 4)])
def test_tiles_of_a_convolution_are_no_taller_than_the_image(conv, H, W, mt):
    assert conv.L.lb_conv3x3(X, 16, 0, WT, None, GX, None, 16, 0, 1, H, W, 16, 16, 1, None) == LB_OK
    assert ["k_conv_tcILi%dE" % mt in c[1] for c in conv.launches("k_conv_tc")] == [True]


@pytest.mark.parametrize("B,H,W,Ci,Co,direct", [(1, 8, 8, 16, 16, True), (1, 75, 100, 64, 96, True), (1, 32, 32, 1024, 256, True),
                                                (1, 9, 3000, 32, 32, True), (2, 64, 64, 512, 512, False),
                                                (1, 1024, 1024, 16, 16, False), (4, 256, 256, 32, 32, False)])
def test_small_forward_layer_is_one_launch_without_scratch(conv, B, H, W, Ci, Co, direct):
    live = conv.L.fake_live()
    args = arguments(conv, "k_conv_tc", ConvArgs)
    conv.L.lb_conv3x3(X, 16, 0, WT, None, GX, None, 16, 0, 1, 8, 8, 16, 16, 1, None)       # the error flag's allocation
    conv.clear()
    del args[:]
    assert conv.L.lb_conv3x3(X, Ci, 0, WT, None, GX, None, Co, 0, B, H, W, Ci, Co, 1, None) == LB_OK
    assert args[0].w == WT and bool(args[0].wp) == (not direct)
    assert len(conv.calls("launch")) == (1 if direct else 2)
    assert [c for c in conv.calls() if "alloc" in c[0].lower()] == [] if direct else conv.L.fake_live() <= live + 1


@pytest.mark.parametrize("Ci,Co,blocks", [(16, 16, 2), (64, 96, 27), (1024, 1024, 1216)])
def test_convolution_starts_beside_the_packing_and_waits_for_it(conv, Ci, Co, blocks):
    # a unit of 16 bytes per thread; the convolution's launch overlaps the packing (w_late: its weights wait)
    args = arguments(conv, "k_conv_tc", ConvArgs)
    assert conv.L.lb_conv3x3_dgrad(GZ, WT, GX, 1, 16, 16, Ci, Co, None) == LB_OK
    assert args[0].w_late == 1 and [c[-1] for c in conv.launches("k_conv_tc")] == ["1"]
    assert [int(c[2]) for c in conv.launches("k_conv_pack")] == [blocks]


def test_scratch_of_the_single_layer_calls_is_given_back_on_request(conv):
    pools = set()
    for dev in (0, 1):
        conv.L.fake_device(dev)
        assert conv.L.lb_conv3x3_wgrad(X, GZ, GW, GB, 1, 9, 40, 32, 16, None) == LB_OK
        pools |= {c[1] for c in conv.calls("cudaMemPoolCreate")}
    conv.clear()
    assert conv.L.lb_conv_release() == LB_OK
    trims = conv.calls("cudaMemPoolTrimTo")
    assert len(trims) == 2 and all(c[2] == "0" for c in trims) and pools <= {c[1] for c in trims}
    conv.fail("cudaMemPoolTrimTo", 1, 700)
    assert conv.L.lb_conv_release() == LB_ECUDA
