"""The collision's launch shapes and the handle's timing calls at the edges
where their kernels or their steps change."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


@pytest.fixture(scope="module")
def H():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2312_14172_gb300 import build, hlbm
    build.build()
    hlbm.load()
    return hlbm


def _fluid(lat, precision):
    """The handle's populations as stored, [blocks, 19, 32]."""
    import torch
    dt, size = (torch.float32, 4) if precision == "fp32" else (torch.float16, 2)
    blocks = sum(-(-b[0] // 32) * b[1] * b[2] for b in lat.boxes)
    return lat.buffer[: blocks * 19 * 32 * size].view(dt).view(blocks, 19, 32)


def _worst(a, b, nx, precision):
    """Largest difference of two such tensors of a box of rows of nx cells, in
    units of the weights; the padding cells of a row's last block hold nothing."""
    import torch
    w = torch.tensor(W, device=a.device)[None, :, None] * (1.0 if precision == "fp32" else 2.0 ** 14)
    last = (nx - 1) // 32
    worst = 0.0
    for k in range(last + 1):
        cells = min(32, nx - 32 * k)
        d = (a[k::last + 1, :, :cells].float() - b[k::last + 1, :, :cells].float()).abs() / w
        worst = max(worst, float(d.max()))
    return worst


def _disturb(lat, precision, seed):
    """Deviations of 1e-3 of the weights in every cell (padding included)."""
    import torch
    v = _fluid(lat, precision)
    g = torch.Generator(device=v.device).manual_seed(seed)
    w = torch.tensor(W, device=v.device)[None, :, None] * (1.0 if precision == "fp32" else 2.0 ** 14)
    for part in v.split(1 << 20):
        part.copy_(1e-3 * w * torch.randn(part.shape, generator=g, device=v.device))
    torch.cuda.synchronize()


@pytest.mark.parametrize("precision,n,bc,particles", [
    ("fp32", (101, 29, 21), 7, 0),       # selects at every wall, a row's single last cell
    ("fp32", (101, 45, 44), 6, 12),
    ("fp16", (70, 33, 30), 0, 0),
    ("fp16", (97, 50, 43), 0, 12),
    ("fp16", (203, 190, 180), 2, 40),    # above twice the L2: blocks prefetch their rows
])
def test_blocks_of_every_height_take_the_same_step(H, precision, n, bc, particles):
    """16 threads (half a warp) to 128 per block, both parities, particles or
    none: the same step.  In FP32 the shapes may differ by rounding (1e-6 of
    the weights); with half storage such a difference can turn a stored value
    to its neighbour, 2^-10 of a deviation of up to 5e-3, here bounded over
    the five steps by 2e-5."""
    import torch
    from paper_2312_14172_gb300 import workloads
    rng = np.random.default_rng(5)
    ref = None
    for shape in ((8, 8, 2), (1, 2, 2), (1, 8, 2), (2, 4, 2), (4, 1, 2)):
        lat = H.Lattice([n + (bc,)], H.make_params(tau=0.7, precision=precision, max_particles=max(1, particles)))
        if particles:
            if ref is None:
                w = workloads.nonspherical(n=n, count=particles, tau=0.7, grid=True)
                P = w["particles"]
                P["U"] = rng.uniform(-1e-3, 1e-3, P["U"].shape)
            lat.add_workload_particles(P)
        _disturb(lat, precision, 7)
        lat.set_launch(*shape)
        lat.step(5)
        lat.sync()
        got = _fluid(lat, precision).clone()
        lat.close()
        if ref is None:
            ref = got
            continue
        assert _worst(ref, got, n[0], precision) <= (1e-6 if precision == "fp32" else 2e-5), shape
    torch.cuda.empty_cache()


def test_autotune_times_the_steps_alone(H):
    """The time per step that the autotuner returns (of twelve steps here) is
    that of the same steps taken again with their graphs there.  Capturing and
    instantiating the two graphs takes longer than the twelve steps of this box
    (44 us of host time against 35 us); a quarter is room for the clock."""
    import torch
    from paper_2312_14172_gb300 import workloads
    w = workloads.single_sphere(n=26, radius=4.0)
    w["particles"] = {k: v[:0] for k, v in w["particles"].items()}
    lat = H.from_workload(w)
    lat.step(8)
    told = lat.autotune(nsteps=3)[3]
    times = []
    for _ in range(9):
        lat.step(2)
        lat.step(12)
        torch.cuda.synchronize()
        lat.step(2)
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record(lat.stream)
        lat.step(12)
        e[1].record(lat.stream)
        torch.cuda.synchronize()
        times.append(e[0].elapsed_time(e[1]) / 12)
    lat.close()
    assert told <= 1.25 * np.median(times)


@pytest.mark.parametrize("contact", [False, True])
@pytest.mark.parametrize("count", [12, 700])
def test_kernel_times_are_those_of_a_steps_kernels(H, count, contact):
    """hlbm_kernel_times launches what hlbm_step launches: the run it leaves
    is that of as many steps, bit for bit, and where the exchange moves few
    particles itself there is no update kernel to time."""
    rng = np.random.default_rng(3)
    n = (100, 90, 80)
    site = rng.permutation(10 * 9 * 8)[:count]
    X = np.stack([site % 10, site // 10 % 9, site // 90], 1) * 10.0 + rng.uniform(4.0, 6.0, (count, 3))
    U = rng.uniform(-1e-3, 1e-3, (count, 3))
    lats = []
    for _ in range(2):
        lat = H.Lattice([n + (0,)], H.make_params(tau=0.7, gravity=(0, 0, -1e-5), max_particles=count))
        lat.add_particles(np.zeros(count, int), np.full((count, 1), 3.0), X, U, U, None, np.full(count, 2.0))
        lat.set_mea_mode("moments")
        if contact:
            lat.set_contact(1e-3, 3.0)
        lat.step(2)
        lats.append(lat)
    a, b = lats
    t = a.kernel_times(3)
    b.step(3)
    sa, sb = a.particle_state(), b.particle_state()
    for k in sa:
        assert np.array_equal(sa[k], sb[k]), k
    assert np.array_equal(a.populations(), b.populations())
    assert t["mea"] > 0.0 and t["collide_stream"] > 0.0
    assert (t["update"] > 0.0) == (contact or count == 700)
    a.close()
    b.close()


@pytest.mark.parametrize("precision,nx,bc", [("fp32", 8192, 6), ("fp16", 16384, 0), ("fp16", 16384, 7)])
@pytest.mark.parametrize("ny,nz,particles", [(6898, 3, 0), (6900, 3, 0), (6898, 7, 2), (6900, 7, 2)])
def test_slices_on_both_sides_of_four_gigabytes(H, precision, nx, bc, ny, nz, particles):
    """A z slice of 6898 such rows ends just below 2^32 bytes, one of 6900 just
    above: odd steps address the one by 32-bit offsets, the other by pointers.
    Both take the step of the one-cell kernel up to rounding (as above, three
    steps) and not its very bits, which would mean that it ran instead.  Without
    particles, and with one at either end of the slices."""
    import torch
    assert (ny * (nx // 32) * 19 * 32 * (4 if precision == "fp32" else 2) > 2 ** 32) == (ny == 6900)
    got = []
    for cells_x in (2, 1):
        lat = H.Lattice([(nx, ny, nz, bc)], H.make_params(tau=0.7, precision=precision, max_particles=2))
        _disturb(lat, precision, 9)
        if particles:
            lat.add_particles([0, 0], [[1.0] * 3] * 2, [[4.3, 2.2, 3.1], [nx - 5.4, ny - 3.3, 3.4]],
                              U=[[1e-3, 2e-3, -1e-3]] * 2, omega=[[1e-3, 0.0, 2e-3]] * 2, rho_p=[2.0, 2.0])
        lat.set_launch(4, 2, cells_x)
        assert lat.get_launch() == (4, 2, cells_x)
        lat.step(3)
        lat.sync()
        got.append(_fluid(lat, precision).clone())
        lat.close()
        del lat
    assert _worst(*got, nx, precision) <= (1e-6 if precision == "fp32" else 2e-5)
    assert not torch.equal(*got)
    del got
    torch.cuda.empty_cache()


@pytest.mark.parametrize("precision,n,count,r,tile_z", [
    ("fp32", (96, 96, 96), 0, 0.0, 2),      # too few blocks for taller bricks
    ("fp16", (96, 96, 96), 50, 5.0, 2),
    ("fp32", (128, 128, 128), 0, 0.0, 2),   # fluid alone
    ("fp32", (128, 128, 128), 20, 6.0, 4),  # particles within twice the L2
    ("fp16", (128, 128, 128), 0, 0.0, 4),
    ("fp16", (160, 160, 160), 1200, 5.0, 4),
    ("fp32", (256, 256, 256), 400, 6.0, 2),   # few candidates, streaming
    ("fp32", (256, 256, 256), 2000, 6.0, 4),  # many
    ("fp16", (256, 256, 256), 0, 0.0, 4),
    ("fp16", (256, 256, 256), 2000, 6.0, 8),
])
def test_default_bricks_follow_size_and_particles(H, precision, n, count, r, tile_z):
    """The default's tile_z is the fastest of 2, 4 and 8 as measured for such
    handles, whether the particles come at once or in two calls; a launch
    shape that was set stays."""
    k = [int(v // (2 * r + 2)) if count else 1 for v in n]
    site = np.arange(count)
    X = (np.stack([site % k[0], site // k[0] % k[1], site // (k[0] * k[1])], 1) + 0.5) * (np.array(n) / k)
    for calls in (1, 2):
        for fixed in (False, True):
            lat = H.Lattice([n + (0,)], H.make_params(precision=precision, max_particles=max(1, count)))
            if fixed:
                lat.set_launch(2, 1, 2)
            for part in np.array_split(site, calls):
                if len(part):
                    lat.add_particles(np.zeros(len(part), int), np.full((len(part), 1), r), X[part],
                                      rho_p=np.full(len(part), 2.0))
            assert lat.get_launch() == ((2, 1, 2) if fixed else (4, tile_z, 2))
            lat.close()


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("n,bc,particles", [
    ((1, 20, 18), 2, 0), ((3, 9, 11), 6, 0), ((31, 18, 17), 4, 0), ((33, 40, 38), 2, 6), ((65, 37, 41), 6, 10),
    ((191, 34, 36), 4, 20), ((193, 34, 36), 4, 20),  # the longest such rows, and longer ones
])
def test_single_ends_between_walls(H, precision, n, bc, particles):
    """Rows that end in a single cell, between walls in y or z: alone such a
    box takes its odd steps by pointers, beside a larger box of even rows by
    32-bit offsets; the same step either way, within rounding as above."""
    rng = np.random.default_rng(n[0])
    k = [max(1, v // 12) for v in n]  # sites 12 cells apart or more, off the walls
    site = rng.permutation(k[0] * k[1] * k[2])[:particles]
    X = (np.stack([site % k[0], site // k[0] % k[1], site // (k[0] * k[1])], 1) + 0.5) * (np.array(n) / k)
    r, U = rng.uniform(3.0, 5.5, (len(site), 1)), rng.uniform(-1e-3, 1e-3, (len(site), 3))
    blocks = -(-n[0] // 32) * n[1] * n[2]
    got = []
    for beside in ([], [(n[0] + 1, n[1] + 1, n[2] + 1, bc)]):
        lat = H.Lattice([n + (bc,)] + beside, H.make_params(tau=0.7, precision=precision, max_particles=max(1, particles)))
        if particles:
            lat.add_particles(np.zeros(len(site), int), r, X, U, U, None, np.full(len(site), 2.0))
        _disturb(lat, precision, 13)
        lat.set_launch(4, 2, 2)
        lat.step(5)
        lat.sync()
        got.append(_fluid(lat, precision)[:blocks].clone())
        lat.close()
    assert _worst(*got, n[0], precision) <= (1e-6 if precision == "fp32" else 2e-5)


def test_a_single_end_costs_little_more_than_a_pair(H):
    """Rows of 33 and of 34 cells take the same blocks, rows and bytes: the
    step of the odd ones, between walls, at most a tenth more."""
    import torch
    took = []
    for nx in (33, 34):
        lat = H.Lattice([(nx, 300, 300, 4)], H.make_params(tau=0.6, precision="fp16", fluid_force=(1e-7, 0, 0)))
        times = []
        for _ in range(7):
            lat.step(16)
            torch.cuda.synchronize()
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record(lat.stream)
            lat.step(16)
            e[1].record(lat.stream)
            torch.cuda.synchronize()
            times.append(e[0].elapsed_time(e[1]))
        took.append(min(times))
        lat.close()
    assert took[0] <= 1.1 * took[1]


@pytest.mark.parametrize("precision,boxes,tile_z", [
    ("fp32", [(32, 32, 32)] * 200, 4), ("fp16", [(32, 32, 32)] * 200, 8),    # many small boxes
    ("fp32", [(128, 128, 128)] * 8, 2), ("fp16", [(128, 128, 128)] * 8, 4),  # few large ones
    ("fp32", [(2000, 3, 2000)], 4), ("fp16", [(2000, 3, 2000)], 8),          # bricks mostly empty in y
])
def test_default_bricks_of_batches_and_thin_boxes(H, precision, boxes, tile_z):
    """As above, fluid alone: the height measured as the fastest of 2, 4 and 8,
    or within 4 % of it and the one that such handles took before."""
    lat = H.Lattice([b + (0,) for b in boxes], H.make_params(precision=precision))
    assert lat.get_launch() == (4, tile_z, 2)
    lat.close()


@pytest.mark.parametrize("precision,few,many", [("fp32", 2, 4), ("fp16", 4, 8)])
def test_default_bricks_with_elongated_particles(H, precision, few, many):
    """Capsules count from half a candidate per tile on."""
    n = (256, 256, 256)
    lat = H.Lattice([n + (0,)], H.make_params(precision=precision, max_particles=400))
    g = np.arange(400)
    X = np.stack([g % 8, g // 8 % 8, g // 64], 1) * 30.0 + 20.0
    lat.add_particles([3] * 100, [[4.0, 4.0, 6.0]] * 100, X[:100], rho_p=[2.0] * 100)
    assert lat.get_launch() == (4, few, 2)
    lat.add_particles([3] * 300, [[4.0, 4.0, 6.0]] * 300, X[100:], rho_p=[2.0] * 300)
    assert lat.get_launch() == (4, many, 2)
    lat.close()
