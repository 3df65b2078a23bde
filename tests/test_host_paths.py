"""Host paths of the library without a GPU, on a stand-in for the CUDA runtime (_fake_cuda.py): the
launches that a call makes, their arguments, and what it copies, waits for and gives back."""
import ctypes
import shutil

import pytest

import _fake_cuda as F

LB_OK, LB_ENOMEM, LB_ECUDA = 0, -3, -4
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
                ("ym", P), ("ldm", I64), ("moff", I32), ("up", P), ("ldu", I64), ("yf2", P)]


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
