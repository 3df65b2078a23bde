"""The tile shapes of lb_step (chosen by the lattice's size) against 32x16 tiles, and rings of every
size class on the node step.

A lattice's fields, nodes and ring readouts do not depend on the tile shape: each case runs once on
its own (8x8, 16x8 or 16x16 tiles by its size) and once as a batch of one with 32x16 tiles, or, in
the 2-byte storage form (which batches do not take), with the warp-strip kernel; bit for bit.  The
lattice sums differ in the order of their partial sums only.
"""
import numpy as np
import pytest

import oracle as O
from paper_2209_14889_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2209_14889_gb300 import lb
    return lb


def _state(s):
    s.sync()
    return s.fields(), s.nodes(), s.series()


def _same(a, b):
    for k in a[0]:
        assert np.array_equal(a[0][k], b[0][k]), k
    assert np.array_equal(a[1], b[1])
    assert np.array_equal(a[2][:, 0], b[2][:, 0]) and np.array_equal(a[2][:, 6:], b[2][:, 6:])
    np.testing.assert_allclose(a[2][:, 1:6], b[2][:, 1:6], rtol=1e-12, atol=1e-12)


TRAP = dict(k=0.05, dx=3.0, dy=0.5, t_eq=30, pull=60, width=30)
CASES = {
    # 8x8 tiles: the smallest lattice, odd sides, a ring across both seams
    "min_8x8": lambda: W.make(8, 8, seed=1),
    "odd_71x53": lambda: W.small(71, 53, seed=2, n_nodes=24, radius=4.0, centre=(1.2, 51.9)),
    # 16x8 tiles: odd and ragged, walls with the trap, sub-steps, the scalar model in a closed box
    "odd_201x117": lambda: W.small(201, 117, seed=3, n_nodes=70, radius=11.0, centre=(199.7, 60.3)),
    "walls_131x150": lambda: W.make(131, 150, rings=[W.ring(60, 9.0, (60.2, 70.7), pull_force=0.0, trap=TRAP)],
                                    seed=4, walls_x=1, walls_y=1),
    "substeps_160x90": lambda: W.small(160, 90, seed=5, n_nodes=40, radius=8.0, Dp=0.6, diffusion_substeps=3),
    "scalar_box_250": lambda: W.make(250, 250, rings=[W.ring(157, 12.5, (74.5, 124.5), pull_force=0.0, trap=TRAP)],
                                     seed=6, walls_x=1, walls_y=1, **W.scalar_physics()),
    # 16x16 tiles
    "even_390x370": lambda: W.small(390, 370, seed=7, n_nodes=64, radius=10.0, centre=(388.0, 3.0)),
    "scalar_660x600": lambda: W.make(660, 600, rings=[W.ring(64, 10.0, (300.2, 3.3))], seed=8, **W.scalar_physics()),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_tile_shapes_match_32x16_tiles_bitwise(case):
    lb = _gpu()
    w = CASES[case]()
    steps = 33
    a, b = lb.Solver.from_workload(w), lb.Solver.from_workload(w)
    a.step(steps)
    batch = lb.Batch([b])
    batch.set_shape(0)
    batch.step(steps)
    batch.sync()
    _same(_state(a), _state(b))
    batch.close()
    a.close()
    b.close()


@pytest.mark.parametrize("nx,ny", [(66, 60), (250, 140)])
def test_tile_shapes_precision_form_match_strip_bitwise(nx, ny):
    lb = _gpu()
    w = W.small(nx, ny, seed=9, n_nodes=40, radius=6.0, centre=(2.4, 30.1))
    a, b = (lb.Solver.from_workload(w, precision=lb.LB_FP16_BF16) for _ in range(2))
    b.set_kernel(lb.LB_KERNEL_STRIP)
    a.step(33)
    b.step(33)
    _same(_state(a), _state(b))
    a.close()
    b.close()


@pytest.mark.parametrize("n_nodes", [3, 31, 256, 257, 1024])
def test_ring_sizes_vs_oracle(n_nodes):
    # one thread per node up to 256 nodes, several nodes per thread beyond (up to the largest ring)
    lb = _gpu()
    r = max(3.0, min(20.0, n_nodes * 0.78 / (2 * np.pi)))
    w = W.make(128, 112, rings=[W.ring(n_nodes, r, (126.3, 50.2), pull_force=1e-3, pull_angle=0.4, trap=TRAP),
                                W.ring(20, 4.0, (30.7, 90.1))], seed=10 + n_nodes)
    s = lb.Solver.from_workload(w)
    s.step(40)
    _, X, ser = _state(s)
    s.close()
    sim = O.Sim.from_workload(w)
    sim.step(40, every=10)
    ref = np.array(sim.series)
    d = X - sim.X
    d -= np.array([128.0, 112.0]) * np.round(d / np.array([128.0, 112.0]))
    # nodes: the FP32 rounding of ~40 displacements of at most ~1e-2; readouts to FP32
    assert np.abs(d).max() <= 1e-6
    for k in range(2):
        c = 6 + 4 * k
        assert np.linalg.norm(ser[:, c:c + 2] - ref[:, c:c + 2]) <= 1e-4 * np.linalg.norm(ref[:, c:c + 2])
        assert np.abs(ser[:, c + 2:c + 4] - ref[:, c + 2:c + 4]).max() <= 1e-6


@pytest.mark.parametrize("n_nodes,radius,trap", [(129, 40.0, False), (192, 12.0, True), (193, 12.0, True), (500, 40.0, True)])
def test_ring_boxes_and_trap_warps_vs_oracle(n_nodes, radius, trap):
    # u(t) on a box too large for shared memory (radius 40) is read from global memory; with the trap
    # the last two of eight warps hold no edge of a ring of up to 192 nodes and advance none of up to 256
    lb = _gpu()
    g = dict(pull_force=0.0, trap=TRAP) if trap else dict(pull_force=1e-3, pull_angle=0.4)
    w = W.make(288, 256, rings=[W.ring(n_nodes, radius, (280.3, 60.2), **g)], seed=20 + n_nodes)
    s = lb.Solver.from_workload(w)
    s.step(40)
    _, X, ser = _state(s)
    s.close()
    sim = O.Sim.from_workload(w)
    sim.step(40, every=10)
    ref = np.array(sim.series)
    d = X - sim.X
    d -= np.array([288.0, 256.0]) * np.round(d / np.array([288.0, 256.0]))
    # as in test_ring_sizes_vs_oracle
    assert np.abs(d).max() <= 1e-6
    assert np.linalg.norm(ser[:, 6:8] - ref[:, 6:8]) <= 1e-4 * np.linalg.norm(ref[:, 6:8])
    assert np.abs(ser[:, 8:10] - ref[:, 8:10]).max() <= 1e-6


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("case", ["odd_71x53", "walls_131x150", "scalar_box_250"])
def test_readout_of_one_field_matches_the_moments_of_all(case, half):
    # a field formed alone, straight into device memory or by way of scratch (host memory, an odd address),
    # is the plane of the pass that forms all three moments (lb_readout_noalloc)
    import ctypes
    lb = _gpu()
    import torch
    w = CASES[case]()
    if half and (w.get("walls_x") or w.get("model")):
        pytest.skip("the 2-byte state takes neither walls nor the scalar model")
    s = lb.Solver.from_workload(w, precision=lb.LB_FP16_BF16 if half else lb.LB_FP32)
    s.step(7)
    noalloc = lb.lib().lb_readout_noalloc
    noalloc.restype = ctypes.c_int
    noalloc.argtypes = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int32]
    for k, fid in lb.FIELDS.items():
        a = s.readout(k).cpu().numpy()
        assert np.array_equal(a, s.readout(k, device=False)), k
        n = a.size * 4
        odd = torch.zeros(n + 8, dtype=torch.uint8, device="cuda")
        assert lb.lib().lb_readout(s.h, fid, ctypes.c_void_p(odd.data_ptr() + 1), n, 1) == 0
        assert np.array_equal(odd[1:1 + n].cpu().numpy().view(np.float32).reshape(a.shape), a), k
        if k in ("drho", "ux", "uy", "Px", "Py"):
            b = torch.zeros(a.shape, dtype=torch.float32, device="cuda")
            assert noalloc(s.h, fid, b.data_ptr(), n, 1) == 0
            assert np.array_equal(b.cpu().numpy(), a), k
    s.close()


@pytest.mark.parametrize("count", [33, 70])
def test_more_rings_than_a_warp_has_lanes_match_the_node_kernel_bitwise(count):
    # beyond 32 rings a tile tests each ring's box by itself, in the gather and in the tail; the same steps with
    # the node step in a launch of its own
    lb = _gpu()
    side = int(np.ceil(np.sqrt(count)))
    rings = [W.ring(12, 2.0, (20.0 * (k % side) + 9.3, 20.0 * (k // side) + 8.6), pull_force=1e-3, pull_angle=0.1 * k)
             for k in range(count)]
    w = W.make(20 * side, 20 * side + 3, rings=rings, seed=12)
    a, b = lb.Solver.from_workload(w), lb.Solver.from_workload(w)
    b.set_node_tail(False)
    a.step(33)
    b.step(33)
    ra, rb = _state(a), _state(b)
    for k in ra[0]:
        assert np.array_equal(ra[0][k], rb[0][k]), k
    assert np.array_equal(ra[1], rb[1]) and np.array_equal(ra[2], rb[2])
    a.close()
    b.close()


@pytest.mark.parametrize("scalar", [False, True])
@pytest.mark.parametrize("nx,ny", [(97, 96), (101, 98), (224, 226), (250, 251), (273, 272), (320, 320), (385, 384)])
def test_tile_shapes_without_rings_match_32x16_tiles_bitwise(nx, ny, scalar):
    # around the limits of the rule without rings: 8x8, 16x8, 32x16 in one wave, 16x16, 32x16
    lb = _gpu()
    w = W.make(nx, ny, seed=11, **(W.scalar_physics() if scalar else {}))
    a, b = lb.Solver.from_workload(w), lb.Solver.from_workload(w)
    a.step(33)
    batch = lb.Batch([b])
    batch.set_shape(0)
    batch.step(33)
    batch.sync()
    _same(_state(a), _state(b))
    batch.close()
    a.close()
    b.close()
