"""GPU kernels and dispatch rules at the sizes where they can go wrong, against the FP64 oracle."""
import numpy as np
import pytest

import oracle as O
from tests import seeded
from tests.test_gpu_parity import L, perturbed, rel  # noqa: F401  (L: the module fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e30])
@pytest.mark.parametrize("q,dims,periodic", [
    (9, (128, 128, 1), 0),   # plain steps in CTAs of one row
    (9, (33, 301, 1), 1),    # of a few rows, a partial CTA at the end
    (9, (700, 303, 1), 2),   # whole CTAs
    (19, (33, 9, 17), 0), (19, (1, 2, 3), 0), (19, (40, 8, 24), 4)])
def test_fp64_pairwise_relaxation(L, q, dims, periodic, scale):  # noqa: F811
    """The FP64 relaxation, which adds the sensor's fractions over common denominators, at densities
    far from 1 too.  A step rounds each population a few times at 2^-53 of its size and K a few
    tens of times at 2^-53 of f / f^neq (about 50 here): 1e-14 and 1e-12 leave a margin of ten."""
    o = O.Oracle(q, *dims, tau=0.83, lid=(0.0, 0.0, 0.0), periodic=periodic)
    f = scale * perturbed(o, seed=17 + sum(dims), amp=0.02)
    lat = L.Lattice(q, *dims, 0.83, dtype=L.LBM_F64, lid=(0.0, 0.0), periodic=periodic)
    lat.set_populations(f)
    L.lbm_set_sensor_field(lat.h, 1)
    lat.step(3)  # two plain steps and a sensor step
    for _ in range(3):
        f, K, _, _ = o.step(f, sensor=True)
    assert rel(lat.populations(), f) <= 1e-14
    assert rel(lat.sensor_field(), K) <= 1e-12
    lat.close()


@pytest.mark.parametrize("dtype", ["LBM_F64", "LBM_F32", "LBM_BF16S"])
@pytest.mark.parametrize("dims,periodic", [((33, 17), 0), ((128, 128), 1), ((700, 302), 2)])
def test_2d_runs_in_graphs_have_the_bits_of_single_steps(L, dims, periodic, dtype):  # noqa: F811
    """A 2-D step's CTAs may start before the step before it has ended: runs of them in graphs, and
    with sensor steps and reads between, must give what steps with a wait after each give."""
    o = O.Oracle(9, *dims, 1, tau=0.7, lid=(0.1, 0.0, 0.0), periodic=periodic)
    f = perturbed(o, seed=5 + sum(dims), amp=0.02)
    import torch

    lats = [L.Lattice(9, *dims, 1, 0.7, dtype=getattr(L, dtype), lid=(0.1, 0.0), periodic=periodic)
            for _ in range(2)]
    for lat in lats:
        lat.set_populations(f)
        L.lbm_set_sensor_every(lat.h, 37)
    L.lbm_set_graphs(lats[1].h, 0)
    for n in (40, 100):
        lats[0].step(n)
        for _ in range(n):
            lats[1].step(1)
            torch.cuda.synchronize()
        assert np.array_equal(lats[0].raw(), lats[1].raw())
        assert np.array_equal(lats[0].sensor(8), lats[1].sensor(8))
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("cin,hidden,batch,h,w,steps", [(3, 8, 2, 12, 13, 1030),  # more than a queue
                                                        (4, 16, 5, 33, 64, 3), (3, 16, 1, 1, 1, 2)])
def test_an_epoch_has_the_bits_of_its_steps(L, cin, hidden, batch, h, w, steps):  # noqa: F811
    """An epoch reads its minibatches from the training set in place and waits once; the same kernels
    on gathered minibatches, a step at a time, give the same losses and parameters."""
    import torch

    g = seeded.rng(cin * 1000 + hidden + steps)
    n = 3 * batch + 1
    X = torch.from_numpy(g.normal(size=(n, cin, h, w)).astype(np.float32)).cuda()
    T = torch.from_numpy(g.normal(size=(n, 1, h, w)).astype(np.float32)).cuda()
    idx = torch.from_numpy(g.integers(0, n, steps * batch).astype(np.int32)).cuda()
    nets = [L.Net(cin, hidden) for _ in range(2)]
    theta = 0.2 * g.normal(size=nets[0].nparam)
    for net in nets:
        net.set_params(theta)
    losses = np.zeros(steps)
    L.lbm_net_train_epoch(nets[0].n, X, T, n, idx, steps, batch, h, w, 1e-3, losses)
    for s in range(steps):
        at = idx[s * batch:(s + 1) * batch].long()
        assert nets[1].train_step(X[at].contiguous(), T[at].contiguous(), 1e-3) == losses[s]
    assert np.array_equal(nets[0].params(), nets[1].params())
    idx[-1] = n  # an index outside is not read, and refused at the end
    with pytest.raises(L.LbmError) as ei:
        L.lbm_net_train_epoch(nets[0].n, X, T, n, idx, steps, batch, h, w, 1e-3, None)
    assert ei.value.status == L.LBM_EINVAL
    for net in nets:
        net.close()


def tag_cases():
    g = seeded.rng(4242)
    sparse = np.zeros((1, 150, 150))
    sparse[0, ::3, ::3] = 1.0  # 2500 boxes: more than come with the first copy, and many rounds
    many = np.zeros((1, 300, 303))
    many[0, ::3, ::3] = 1.0  # 10100 boxes: more than the device's queues hold
    long = np.zeros((1, 20, 9000))  # a tag grid too long for the device's signatures
    long[0, 3:9, g.integers(0, 9000, 30)] = 1.0
    wide = (g.random((1, 130, 2050)) < 0.002).astype(float)
    solid = (g.random((33, 18, 65)) < 0.03).astype(float)
    last = np.zeros((40, 1, 1), dtype=float)
    last[39] = 1.0
    return {"sparse": (sparse, 1, 0), "many": (many, 1, 0), "long": (long, 1, 0),
            "wide": (wide, 1, 1), "solid": (solid, 1, 0), "solid_w3": (solid, 3, 1), "last": (last, 1, 0)}


@pytest.mark.parametrize("name", ["sparse", "many", "long", "wide", "solid", "solid_w3", "last"])
def test_regrid_on_the_device_and_on_the_host(L, name):  # noqa: F811
    """Clustering at the limits of the device's queues and beyond them, where the host takes over;
    the buffers a handle keeps serve a second, different regrid.  Boxes and tags are whole numbers."""
    import torch

    from oracle import regrid as R

    K, w, buffer = tag_cases()[name]
    nz, ny, nx = K.shape
    lat = L.Lattice(L.LBM_D3Q19 if nz > 1 else L.LBM_D2Q9, nx, ny, nz, 0.6, dtype=L.LBM_F64)
    for field in (K, K[:, ::-1].copy(), K):
        ref_boxes, ref_tags = R.regrid(field, 0.5, coarsen=1, buffer=buffer, efficiency=0.9, min_width=w)
        boxes, tags = lat.regrid(0.5, coarsen=1, buffer=buffer, efficiency=0.9, min_width=w,
                                 field=torch.from_numpy(field).cuda())
        assert np.array_equal(tags, ref_tags)
        assert boxes.tolist() == ref_boxes.tolist()
    lat.close()


@pytest.mark.parametrize("dtype", ["LBM_F32", "LBM_F16S", "LBM_BF16S"])
@pytest.mark.parametrize("dims,periodic", [((1, 725, 724), 0), ((33, 180, 90), 5), ((99, 80, 80), 0),
                                           ((257, 3, 681), 3), ((5000, 2, 53), 4), ((33, 180, 80), 7)])
def test_3d_steps_in_a_line_have_the_bits_of_rows(L, dims, periodic, dtype):  # noqa: F811
    """Sensor steps that take a plane's cells in a line, whose CTAs share tiles (from 2^19 cells on, the
    last case below), against the allocation-free call, which keeps to rows: populations and maxima, with
    the tile buffers alternating."""
    import torch

    nx, ny, nz = dims
    o = O.Oracle(19, *dims, tau=0.7, lid=(0.1, 0.0, 0.02), periodic=periodic)
    lat = L.Lattice(19, *dims, 0.7, dtype=getattr(L, dtype), lid=(0.1, 0.02), periodic=periodic)
    lat.set_populations(perturbed(o, seed=7 + sum(dims), amp=0.02))
    L.lbm_set_sensor_every(lat.h, 1)
    src = torch.from_numpy(lat.raw().copy()).cuda()
    dst = torch.empty_like(src)
    maxima = torch.empty(L.lbm_nblocks(lat.h, 8), dtype=torch.float64, device="cuda")
    for _ in range(4):
        lat.step(1)
        L.lbm_step_noalloc(19, getattr(L, dtype), nx, ny, nz, 0.7, 0.1, 0.02, periodic, src, dst, 8, maxima,
                           torch.cuda.current_stream())
        torch.cuda.synchronize()
        assert np.array_equal(lat.raw(), dst.cpu().numpy())
        assert np.array_equal(lat.sensor(8), maxima.cpu().numpy())
        src, dst = dst, src
    lat.close()


@pytest.mark.parametrize("dtype", ["LBM_F64", "LBM_F32", "LBM_F16S", "LBM_BF16S"])
@pytest.mark.parametrize("q,dims,periodic", [(19, (99, 80, 80), 0), (19, (98, 80, 80), 5), (19, (2, 600, 440), 0),
                                             (19, (256, 3, 683), 2), (19, (9, 7, 33), 7), (9, (45, 61, 1), 0),
                                             (9, (33, 1, 1), 0), (9, (700, 3, 1), 3)])
def test_plain_steps_in_a_line_match_the_oracle(L, q, dims, periodic, dtype):  # noqa: F811
    """Plain steps over a plane's cells in a line, one and two cells a lane, at sides where rows, faces
    and the last warp end anywhere.  Two steps round a population a few times at the type's precision
    relative to the largest one (16-bit types: that of f - w, here under 0.1 of it)."""
    o = O.Oracle(q, *dims, tau=0.8, lid=(0.1, 0.0, 0.0), periodic=periodic)
    lat = L.Lattice(q, *dims, 0.8, dtype=getattr(L, dtype), lid=(0.1, 0.0), periodic=periodic)
    lat.set_populations(perturbed(o, seed=3 + sum(dims), amp=0.02))
    f = lat.populations()  # as stored
    L.lbm_set_sensor_every(lat.h, 1000)
    lat.step(2)
    for _ in range(2):
        f, _, _, _ = o.step(f, sensor=False)
    assert rel(lat.populations(), f) <= {"LBM_F64": 1e-14, "LBM_F32": 2e-6, "LBM_F16S": 2e-4, "LBM_BF16S": 2e-3}[dtype]
    lat.close()


@pytest.mark.parametrize("name", ["boxes_w2", "rows"])
def test_regrid_beyond_the_queues_while_other_work_runs(L, name):  # noqa: F811
    """Rounds that outgrow the device's queues: more than 8192 boxes of width 2 in a round, and rows whose signatures
    outgrow the pool.  Steps of another lattice hold the SMs, so that CTAs of one launch start at
    different times, before and after one of them finds a queue full; the boxes are the host's."""
    import torch

    from oracle import regrid as R

    if name == "rows":
        K, w = np.zeros((1, 1500, 1500)), 1
        K[0, ::3] = 1.0
    else:
        K, w = np.zeros((1, 650, 655)), 2
        K[0, ::5, ::5] = K[0, 1::5, ::5] = K[0, ::5, 1::5] = K[0, 1::5, 1::5] = 1.0
    ref_boxes, ref_tags = R.regrid(K, 0.5, coarsen=1, buffer=0, efficiency=0.9, min_width=w)
    assert name == "rows" or len(ref_boxes) > 8192
    lat = L.Lattice(L.LBM_D2Q9, K.shape[2], K.shape[1], 1, 0.6, dtype=L.LBM_F64)
    field = torch.from_numpy(K).cuda()
    side = torch.cuda.Stream()
    other = L.Lattice(L.LBM_D3Q19, 128, 128, 128, 0.6, dtype=L.LBM_F32, stream=side)
    for _ in range(3):
        other.step(200)
        boxes, tags = lat.regrid(0.5, coarsen=1, buffer=0, efficiency=0.9, min_width=w, field=field)
        assert np.array_equal(tags, ref_tags)
        assert boxes.tolist() == ref_boxes.tolist()
    side.synchronize()
    other.close()
    lat.close()


@pytest.mark.parametrize("w", [9, 66, 8193, 2 ** 31 - 31, 2 ** 31 - 1])
def test_regrid_with_pieces_wider_than_the_grid(L, w):  # noqa: F811
    """A least width that few or no cuts leave, up to the largest int: one box, or the oracle's few."""
    import torch

    from oracle import regrid as R

    K = (seeded.rng(99).random((33, 18, 65)) < 0.03).astype(float)
    lat = L.Lattice(L.LBM_D3Q19, 65, 18, 33, 0.6, dtype=L.LBM_F64)
    ref_boxes, ref_tags = R.regrid(K, 0.5, coarsen=1, buffer=0, efficiency=0.9, min_width=w)
    assert (len(ref_boxes) == 1) == (w > 9)
    boxes, tags = lat.regrid(0.5, coarsen=1, buffer=0, efficiency=0.9, min_width=w,
                             field=torch.from_numpy(K).cuda())
    assert np.array_equal(tags, ref_tags)
    assert boxes.tolist() == ref_boxes.tolist()
    lat.close()


@pytest.mark.parametrize("dtype", ["LBM_F64", "LBM_F32", "LBM_F16S", "LBM_BF16S"])
@pytest.mark.parametrize("nx,ny", [(33, 17), (700, 303)])
def test_2d_slab_steps_read_the_halos_just_filled(L, nx, ny, dtype):  # noqa: F811
    """A 2-D slab that is its own neighbour, its halos filled from the device by the launch before each
    step and nothing waited for: the bits of a lattice that is periodic along the cut axis."""
    import torch

    o = O.Oracle(9, nx, ny, 1, tau=0.7, lid=(0.0, 0.0, 0.0), periodic=2)
    f = perturbed(o, seed=11 + nx, amp=0.02)
    whole, slab = [L.Lattice(9, nx, ny, 1, 0.7, dtype=getattr(L, dtype), lid=(0.0, 0.0), periodic=p)
                   for p in (2, 0)]
    slab.set_halo(L.LBM_HALO_LO | L.LBM_HALO_HI)
    for lat in (whole, slab):
        L.lbm_set_kernel_variant(lat.h, L.LBM_KERNEL_CELL)
        L.lbm_set_sensor_every(lat.h, 7)
        lat.set_populations(f)
    up, down = [torch.empty(L.lbm_halo_size(slab.h)[1], dtype=torch.uint8, device="cuda") for _ in range(2)]
    for _ in range(50):
        L.lbm_halo_export(slab.h, L.LBM_HALO_HI, up)
        L.lbm_halo_export(slab.h, L.LBM_HALO_LO, down)
        L.lbm_halo_import(slab.h, L.LBM_HALO_LO, up)
        L.lbm_halo_import(slab.h, L.LBM_HALO_HI, down)
        slab.step(1)
        whole.step(1)
    assert np.array_equal(slab.raw(), whole.raw())
    assert np.array_equal(slab.sensor(8), whole.sensor(8))
    for lat in (whole, slab):
        lat.close()


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("q,dims,c5", [(9, (40, 33, 1), (1, 1, 0)), (19, (20, 17, 24), (0, 0, 1))])
def test_fp64_nan_maxima_stand_out(L, q, dims, c5, value):  # noqa: F811
    """One infinite or NaN population makes K NaN, of either sign, in the cell it arrives at: its block's
    maximum is NaN and flagged, the others are those of a run without it."""
    o = O.Oracle(q, *dims, tau=0.7, lid=(0.0, 0.0, 0.0))
    f = perturbed(o, seed=41, amp=0.02)
    lat = L.Lattice(q, *dims, 0.7, dtype=L.LBM_F64, lid=(0.0, 0.0))
    maxima = []
    x, y, z = (n // 2 for n in dims)
    for v in (f[5, z, y, x], value):
        f[5, z, y, x] = v
        lat.set_populations(f)
        lat.step(1)
        maxima.append(lat.sensor(8).reshape([-(-n // 8) for n in dims[::-1]]))
    hit = np.zeros_like(maxima[0], dtype=bool)
    hit[(z + c5[2]) // 8, (y + c5[1]) // 8, (x + c5[0]) // 8] = True
    assert np.array_equal(np.isnan(maxima[1]), hit)
    assert np.array_equal(maxima[1][~hit], maxima[0][~hit])
    assert lat.flag(1e300, block=8).reshape(hit.shape)[hit] > 0
    lat.close()


@pytest.mark.parametrize("scale", [1e50, 1e90, 1e140])
@pytest.mark.parametrize("q,dims", [(9, (128, 33, 1)), (19, (33, 9, 17))])
def test_fp64_sensor_at_any_density(L, q, dims, scale):  # noqa: F811
    """K does not change with the scale of the populations, however far their products of several are out
    of range.  The tolerance is that of test_fp64_pairwise_relaxation."""
    o = O.Oracle(q, *dims, tau=0.83, lid=(0.0, 0.0, 0.0))
    f = scale * perturbed(o, seed=19, amp=0.02)
    lat = L.Lattice(q, *dims, 0.83, dtype=L.LBM_F64, lid=(0.0, 0.0))
    lat.set_populations(f)
    L.lbm_set_sensor_field(lat.h, 1)
    lat.step(1)
    _, K, _, _ = o.step(f, sensor=True)
    assert np.isfinite(K).all()
    assert rel(lat.sensor_field(), K) <= 1e-12
    lat.close()


@pytest.mark.parametrize("scale", [1e160, 1e300])
@pytest.mark.parametrize("q,dims", [(9, (128, 33, 1)), (19, (33, 9, 17))])
def test_fp64_populations_at_any_density(L, q, dims, scale):  # noqa: F811
    """No square of a momentum leaves the range before its populations do.  Tolerances as in
    test_fp64_pairwise_relaxation."""
    o = O.Oracle(q, *dims, tau=0.83, lid=(0.0, 0.0, 0.0))
    f = scale * perturbed(o, seed=23, amp=0.02)
    lat = L.Lattice(q, *dims, 0.83, dtype=L.LBM_F64, lid=(0.0, 0.0))
    lat.set_populations(f)
    L.lbm_set_sensor_field(lat.h, 1)
    lat.step(3)  # two plain steps and a sensor step
    for _ in range(3):
        f, K, _, _ = o.step(f, sensor=True)
    assert rel(lat.populations(), f) <= 1e-14
    assert rel(lat.sensor_field(), K) <= 1e-12
    lat.close()


@pytest.mark.parametrize("dtype,nx,ny", [("LBM_F64", 320, 320), ("LBM_F64", 384, 380), ("LBM_F64", 416, 416),
                                         ("LBM_F32", 448, 448), ("LBM_F32", 480, 480), ("LBM_F32", 333, 444),
                                         ("LBM_F16S", 448, 450), ("LBM_F16S", 900, 900)])
def test_2d_steps_of_any_share_of_the_gpu_overlap(L, dtype, nx, ny):  # noqa: F811
    """Steps that fill the SMs in part, just or more than once let the next one start early or late: runs,
    with the sensor at every third step, give the bits of steps with a wait after each."""
    import torch

    o = O.Oracle(9, nx, ny, 1, tau=0.7, lid=(0.1, 0.0, 0.0))
    f = perturbed(o, seed=nx + ny, amp=0.02)
    lats = [L.Lattice(9, nx, ny, 1, 0.7, dtype=getattr(L, dtype), lid=(0.1, 0.0)) for _ in range(2)]
    for lat in lats:
        lat.set_populations(f)
        L.lbm_set_graphs(lat.h, 0)
    for every in (3, 1000):
        for lat in lats:
            L.lbm_set_sensor_every(lat.h, every)
        lats[0].step(30)
        for _ in range(30):
            lats[1].step(1)
            torch.cuda.synchronize()
        assert np.array_equal(lats[0].raw(), lats[1].raw())
        assert np.array_equal(lats[0].sensor(8), lats[1].sensor(8))
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("dtype", ["LBM_F32", "LBM_F16S"])
def test_sensor_steps_replayed_from_a_callers_graph(L, dtype):  # noqa: F811
    """A plain and a sensor step in a caller's graph, replayed with steps outside it between: each
    sensor step's maxima are its own, not those of an earlier one in the same buffer."""
    import torch

    dims = (81, 90, 75)  # ragged rows, over 2^19 cells: a line outside graphs
    o = O.Oracle(19, *dims, tau=0.7, lid=(0.0, 0.0, 0.0))
    f = perturbed(o, seed=61, amp=0.05)  # decays from step to step
    side = torch.cuda.Stream()
    a, b = [L.Lattice(19, *dims, 0.7, dtype=getattr(L, dtype), lid=(0.0, 0.0), stream=side) for _ in range(2)]
    for lat in (a, b):
        lat.set_populations(f)
        lat.step(2)
    out = torch.empty(L.lbm_nblocks(a.h, 8), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        a.step(2)
        L.lbm_sensor_dev(a.h, 8, out)
    for k in range(6):
        if k % 3 == 2:
            a.step(2)
            got = a.sensor(8)
        else:
            with torch.cuda.stream(side):
                graph.replay()
            torch.cuda.synchronize()
            got = out.cpu().numpy()
        b.step(2)
        assert np.array_equal(got, b.sensor(8)), k
    assert np.array_equal(a.raw(), b.raw())
    for lat in (a, b):
        lat.close()
