"""The kernels that AUTO picks for each kind of step against the generic ones.

Widths that are no multiple of 4 (the z-marching kernels with plain row
prefetches), steps with the flow off (the Heun kernels on the Q mirror) and
Gauss-Seidel coupling (the LB halves of the z-marching kernels, then the Heun
kernels with the new velocity), with and without walls, on shapes with ragged
tiles in x and y, several tiles and z-chunks, and the smallest width; then what
reads the state the kernels leave, the graphs that replay them, and the
convolutions over many plane pairs.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (nz, ny, nx): one partial tile, several with a ragged last one, rows of every
# alignment of a 16-byte group, fewer planes than a chunk, the smallest width
SHAPES = [(9, 11, 5), (37, 19, 45), (21, 9, 101), (1, 3, 66), (2, 17, 35), (6, 40, 4)]


@pytest.fixture(scope="module")
def lcbp():
    import torch
    from paper_0901_3293_gb300 import build
    build.build()
    from paper_0901_3293_gb300 import lcbp as L
    torch.cuda.set_device(0)
    return L


def pair(L, shape, dtype, mode):
    """Two lattices in the same state (BPII with noise), AUTO and GENERIC."""
    nz, ny, nx = shape
    out = []
    for path in (L.PATH_AUTO, L.PATH_GENERIC):
        lat = L.Lattice(nx, ny, nz, dtype=dtype).set_path(path)
        lat.set_flow(flow_on="noflow" not in mode, coupling=L.GAUSS_SEIDEL if "seidel" in mode else L.JACOBI)
        if "walls" in mode:
            lat.set_walls(True, (0.2, 0.0, 0.0, -0.1, 0.0))
        lat.init_q(L.BPII, 0.3, noise=1e-3, seed=4)
        if "noflow" not in mode:
            lat.init_f_equilibrium(1.0)
        out.append(lat)
    return out


# FP64: rounding of O(1/2) fields over 10 steps (as the parity tests take it).
# FP32: the bounds of the fast-against-generic comparison of the parity tests.
TOL = {"f64": (1e-13, 1e-14), "f32": (1e-6, 1e-8)}


def check(L, shape, dtype, mode, steps):
    a, b = pair(L, shape, dtype, mode)
    for lat in (a, b):
        lat.step(steps)
    tq, tu = TOL[dtype]
    assert np.abs(a.read_q() - b.read_q()).max() < tq
    if "noflow" not in mode:
        assert np.abs(a.read_u() - b.read_u()).max() < tu
        assert np.abs(a.read_f() - b.read_f()).max() <= (2.0 ** -23 if dtype == "f32" else tq)


@pytest.mark.parametrize("mode", ["flow", "walls"])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape", SHAPES)
def test_marching_kernels_match_generic(lcbp, shape, dtype, mode):
    check(lcbp, shape, dtype, mode, 11)


# grids large enough for the marching kernels where short ones stay generic: several waves
# of 32-wide tiles, narrow tiles (13 wide), widths of 17 to 23, and shapes on both
# sides of the line
@pytest.mark.parametrize("mode", ["flow", "walls", "seidel"])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape", [(37, 47, 45), (60, 9, 101), (70, 85, 13), (112, 70, 19), (21, 40, 33), (50, 50, 18)])
def test_larger_odd_widths_match_generic(lcbp, shape, dtype, mode):
    if mode == "seidel" and dtype == "f32":
        pytest.skip("FP32 Gauss-Seidel: by its rounding errors below")
    check(lcbp, shape, dtype, mode, 6)


# every shape above: AUTO leaves some of them to the generic kernels, FAST1 none
@pytest.mark.parametrize("mode", ["flow", "walls", "seidel", "seidel_walls"])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape", SHAPES + [(70, 85, 13), (112, 70, 19), (21, 40, 33), (50, 50, 18), (48, 65, 80)])
def test_marching_kernels_forced(lcbp, shape, dtype, mode):
    """FAST1 against GENERIC, whichever AUTO would take, and the kernels of a step counted on both sides; FP32
    Gauss-Seidel by its rounding errors (as below)."""
    a, b = pair(lcbp, shape, dtype, mode)
    a.set_path(lcbp.PATH_FAST1)
    exact = pair(lcbp, shape, "f64", mode)[1] if dtype == "f32" and "seidel" in mode else None
    assert len(a.profile_steps(6)) == (4 if "seidel" in mode else 2)
    assert len(b.profile_steps(6)) == (5 if "seidel" in mode else 3)
    if exact is not None:
        exact.step(6)
        for read in ("read_q", "read_u", "read_f"):
            want = getattr(exact, read)()
            mine, theirs = (np.linalg.norm(getattr(lat, read)() - want) for lat in (a, b))
            assert mine <= 2 * theirs
        return
    tq, tu = TOL[dtype]
    assert np.abs(a.read_q() - b.read_q()).max() < tq
    assert np.abs(a.read_u() - b.read_u()).max() < tu
    assert np.abs(a.read_f() - b.read_f()).max() <= (2.0 ** -23 if dtype == "f32" else tq)


@pytest.mark.parametrize("dtype,mode,shape,kernels", [
    ("f32", "flow", (9, 11, 5), 2), ("f32", "flow", (37, 47, 45), 2), ("f32", "flow", (50, 50, 18), 3),
    ("f32", "flow", (70, 85, 13), 2), ("f32", "flow", (9, 200, 100), 2), ("f32", "walls", (37, 19, 45), 2),
    ("f64", "flow", (70, 85, 13), 3), ("f64", "flow", (37, 19, 45), 2), ("f32", "seidel", (48, 64, 80), 4),
    ("f32", "seidel", (50, 100, 20), 5), ("f64", "seidel", (21, 40, 33), 4), ("f32", "noflow", (9, 11, 5), 2),
    ("f32", "flow", (9, 11, 3), 3), ("f32", "flow", (500, 1, 45), 3), ("f64", "flow", (500, 1, 45), 3),
    ("f32", "flow", (1000, 2, 25), 3), ("f32", "flow", (600, 5, 41), 2), ("f32", "seidel", (3000, 1, 32), 5),
    ("f32", "flow", (2000, 3, 33), 3), ("f64", "flow", (2000, 2, 45), 3), ("f64", "seidel", (1000, 2, 25), 4),
    ("f32", "flow", (3000, 5, 17), 3), ("f32", "seidel", (1, 512, 512), 5)])
def test_kernels_that_auto_picks(lcbp, dtype, mode, shape, kernels):
    """Both sides of the size rules: 2 marching or Heun kernels a step, 4 with Gauss-Seidel; 3 and 5 generic ones."""
    assert len(pair(lcbp, shape, dtype, mode)[0].profile_steps(1)) == kernels


# 128 positions per CTA: one partly filled CTA, several, a width of 32 lanes; the
# longest chunk (16 planes) with a shorter last one
@pytest.mark.parametrize("mode", ["noflow", "noflow_walls"])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape", [(3, 5, 4), (1, 11, 13), (37, 19, 45), (8, 16, 32), (50, 160, 250)])
def test_heun_kernels_match_generic(lcbp, shape, dtype, mode):
    check(lcbp, shape, dtype, mode, 10)


# planes far smaller than a CTA: FP64 takes the sites of all planes in one sequence at
# every shape, FP32 in long lattices (the last CTA of each partly filled; one chunk of several planes and a shorter last one)
@pytest.mark.parametrize("mode", ["noflow", "noflow_walls", "seidel"])
@pytest.mark.parametrize("dtype,shape", [("f64", (7, 1, 5)), ("f64", (130, 5, 7)), ("f32", (4100, 5, 5)),
                                         ("f32", (4999, 8, 17)), ("f32", (9000, 1, 4))])
def test_heun_kernels_in_thin_lattices(lcbp, dtype, shape, mode):
    if mode == "seidel" and dtype == "f32":
        pytest.skip("FP32 Gauss-Seidel: by its rounding errors below")
    check(lcbp, shape, dtype, mode, 6)


@pytest.mark.parametrize("shape,kernels", [((300, 300, 5), 2), ((350, 350, 5), 3), ((16384, 4, 4), 3), ((340, 350, 8), 2),
                                           ((500, 500, 8), 3), ((500, 500, 12), 2), ((26000, 3, 12), 3)])
def test_heun_kernels_where_they_pay(lcbp, shape, kernels):
    """Flow off, FP32: two Heun kernels a step, but the generic three where the mirror's rows are too many for their
    few sites (there the two took up to 1.8 times as long)."""
    lat = lcbp.Lattice(shape[2], shape[1], shape[0]).set_flow(flow_on=False).init_q(lcbp.BPII, 0.3, noise=1e-3, seed=4)
    assert len(lat.profile_steps(1)) == kernels
    wide = lcbp.Lattice(shape[2], shape[1], shape[0] // 100, dtype="f64").set_flow(flow_on=False)
    assert len(wide.init_q(lcbp.BPII, 0.3, seed=4).profile_steps(1)) == 2


def test_flow_switched_on_after_relaxation(lcbp):
    """The state moves between the kernel sets with its mirrors' images intact."""
    a, b = pair(lcbp, (12, 10, 36), "f64", "noflow")
    for lat in (a, b):
        lat.step(5)
        lat.set_flow(flow_on=True).init_f_equilibrium(1.0).step(3)
        lat.set_flow(flow_on=False).step(3)
        lat.set_flow(flow_on=True).step(2)
    assert np.abs(a.read_q() - b.read_q()).max() < 1e-13
    assert np.abs(a.read_u() - b.read_u()).max() < 1e-14


GS_SHAPES = [(9, 11, 5), (13, 18, 64), (37, 19, 45), (1, 3, 66), (2, 17, 36)]


@pytest.mark.parametrize("mode", ["seidel", "seidel_walls"])
@pytest.mark.parametrize("shape", GS_SHAPES)
def test_gauss_seidel_matches_generic(lcbp, shape, mode):
    check(lcbp, shape, "f64", mode, 11)


@pytest.mark.parametrize("mode", ["seidel", "seidel_walls"])
@pytest.mark.parametrize("shape", GS_SHAPES)
def test_gauss_seidel_f32_rounds_like_generic(lcbp, shape, mode):
    """FP32 against the generic FP64 run: both FP32 kernel sets do the same operations per site in another
    order, so their rounding errors are of one size (2-norms within a factor of two)."""
    a, b = pair(lcbp, shape, "f32", mode)
    exact = pair(lcbp, shape, "f64", mode)[1]
    for lat in (a, b, exact):
        lat.step(11)
    for read in ("read_q", "read_u", "read_f"):
        want = getattr(exact, read)()
        mine, theirs = (np.linalg.norm(getattr(lat, read)() - want) for lat in (a, b))
        assert mine <= 2 * theirs


def test_coupling_switched_between_steps(lcbp):
    a, b = pair(lcbp, (12, 10, 12), "f64", "flow")
    for lat in (a, b):
        lat.step(4)
        lat.set_flow(coupling=lcbp.GAUSS_SEIDEL).step(3)
        lat.set_flow(coupling=lcbp.JACOBI).step(4)
    assert np.abs(a.read_q() - b.read_q()).max() < TOL["f64"][0]
    assert np.abs(a.read_u() - b.read_u()).max() < TOL["f64"][1]


@pytest.mark.parametrize("mode", ["flow", "walls"])
@pytest.mark.parametrize("shape", [(30, 33, 16), (21, 18, 12), (5, 100, 13)])
def test_narrow_tiles_match_generic(lcbp, shape, mode):
    """Lattices at most 16 wide: 16 x 16 tiles, full and ragged in x and y."""
    check(lcbp, shape, "f32", mode, 11)


# dtype, mode, shape: every kernel set, the graphs of 16 and 2 steps and single steps
@pytest.mark.parametrize("dtype,mode,shape", [("f32", "flow", (24, 16, 40)), ("f32", "walls", (17, 9, 37)),
                                              ("f64", "flow", (6, 10, 36)), ("f32", "noflow", (9, 16, 24)),
                                              ("f32", "seidel", (10, 12, 36))])
@pytest.mark.parametrize("before", [0, 1])
def test_long_runs_equal_single_steps(lcbp, dtype, mode, shape, before):
    """The same kernels in the same order, whichever graphs replay them and from
    whichever of the two population buffers: equal to the bit."""
    a = pair(lcbp, shape, dtype, mode)[0]
    b = pair(lcbp, shape, dtype, mode)[0]
    for lat in (a, b):
        lat.step(before)
    a.step(51)
    for _ in range(51):
        b.step(1)
    assert np.array_equal(a.read_q(), b.read_q())
    if mode != "noflow":
        assert np.array_equal(a.read_u(), b.read_u())
        assert np.array_equal(a.read_f(), b.read_f())


@pytest.mark.parametrize("dtype,mode", [("f32", "flow"), ("f32", "seidel"), ("f64", "flow"), ("f32", "noflow")])
def test_runs_between_parameter_changes_equal_single_steps(lcbp, dtype, mode):
    """Changes of a parameter drop the graphs, runs of every length follow: those that replay graphs of two steps and
    those that capture graphs of 16, at once or when enough steps have gone by."""
    a = pair(lcbp, (10, 12, 36), dtype, mode)[0]
    b = pair(lcbp, (10, 12, 36), dtype, mode)[0]
    for k, runs in enumerate([(1, 16), (47,), (48, 2), (17, 17, 17, 16), (128,)]):
        for lat in (a, b):
            lat.set_ldg(0.01, 3.1, 0.01 + 1e-4 * k, 2 * np.pi / 16)
        for n in runs:
            a.step(n)
        for _ in range(sum(runs)):
            b.step(1)
    assert np.array_equal(a.read_q(), b.read_q())
    if mode != "noflow":
        assert np.array_equal(a.read_f(), b.read_f())


def test_runs_between_parameter_changes_capture_no_long_graph(lcbp):
    """A run of 40 Gauss-Seidel steps after a change of a parameter takes no longer than the same steps in two runs of
    20, which are too short for the graph of 16 steps (a quarter more, were it captured)."""
    import time

    def seconds(lat, runs):
        best = np.inf
        for k in range(25):
            lat.set_ldg(0.01, 3.1, 0.01 + 1e-6 * k, 2 * np.pi / 16)
            lat.synchronize()
            t0 = time.perf_counter()
            for n in runs:
                lat.step(n)
            lat.synchronize()
            best = min(best, time.perf_counter() - t0)
        return best

    lat = pair(lcbp, (32, 32, 32), "f32", "seidel")[0]
    lat.step(2)
    assert seconds(lat, (40,)) < 1.1 * seconds(lat, (20, 20))


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("mode", ["flow", "walls", "noflow"])
@pytest.mark.parametrize("shape", [(7, 9, 33), (6, 12, 64), (1, 5, 5)])
def test_device_reads_and_diagnostics_from_the_mirrors(lcbp, shape, dtype, mode):
    """After a step Q and rho u live in the padded mirrors.  Reads into device
    tensors equal the host's to the bit; the diagnostics of Q equal those of the same
    field held flat by a generic lattice but for the order of their FP64 sums (1e-12
    of the sum of n terms of one size)."""
    import torch
    lat = pair(lcbp, shape, dtype, mode)[0]
    lat.step(3)
    diag = lat.free_energy(), lat.defect_fraction()
    nptype = np.float32 if dtype == "f32" else np.float64
    for read, comps in (("read_q", 5), ("read_u", 3), ("read_rho", 1)):
        host = getattr(lat, read)(dtype=nptype)
        out = torch.empty(host.shape, device="cuda", dtype=torch.float32 if dtype == "f32" else torch.float64)
        getattr(lat, read)(out=out)
        assert np.array_equal(out.cpu().numpy(), host)
    flat = pair(lcbp, shape, dtype, mode)[1]
    flat.set_q(lat.read_q())
    want = flat.free_energy(), flat.defect_fraction()
    assert abs(diag[0] - want[0]) <= 1e-12 * max(1.0, abs(want[0]))
    assert diag[1] == want[1]


# planes much smaller than a CTA and slightly larger ones, one chunk and many, chunks that straddle CTAs
@pytest.mark.parametrize("dtype,tol", [("f64", 1e-12), ("f32", 1e-4)])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("shape", [(50, 1, 4), (1500, 5, 7), (11, 17, 16), (3, 1, 300), (640, 20, 9)])
def test_diagnostics_of_thin_lattices(lcbp, shape, walls, dtype, tol):
    """Against the oracle, from the flat field and from the mirrors that a step leaves: F with the bounds of the other
    energy tests, whole counts of defects (the threshold in a gap of the eigenvalues), the mass to FP32 moments."""
    from oracle import lbq
    p = lbq.Params(walls_z=walls, q_wall=(0.2, 0.0, 0.0, -0.1, 0.0)) if walls else lbq.Params()
    lat = lcbp.Lattice(shape[2], shape[1], shape[0], dtype=dtype)
    lat.set_ldg(p.A0, p.gamma, p.K, p.q0).set_flow(p.tau_f, p.xi, p.Gamma)
    if walls:
        lat.set_walls(True, p.q_wall)
    lat.init_q(lcbp.BPII, 0.3, noise=1e-3, seed=4).init_f_equilibrium(1.0)
    for _ in range(2):
        Q = lbq.q5_to_q9(lat.read_q())
        F = lbq.free_energy(Q, p)
        assert abs(lat.free_energy() - F) < tol * max(1.0, abs(F))
        top = np.sort(np.linalg.eigvalsh(Q)[..., 2], axis=None)
        mid = top.size // 4 + np.argmax(np.diff(top[top.size // 4: 3 * top.size // 4]))
        assert lat.defect_fraction(float(top[mid] + top[mid + 1]) / 2) * lat.n == mid + 1
        mass = lat.read_f().sum()
        assert abs(lat.totals()[0] - mass) < (1e-12 if dtype == "f64" else 2.0 ** -23) * mass
        lat.step(1)


@pytest.mark.parametrize("dtype,dims", [("f32", (32, 32, 36)), ("f32", (101, 75, 66)), ("f64", (33, 40, 22))])
def test_first_step_tunes_within_a_short_run(lcbp, dtype, dims):
    """The tuning that the first step of a shape waits for takes at most as long as 700 steps of the shape (some 20
    candidates, a few launches each, the slowest at several times the best; measured 50 to 280)."""
    import time

    def seconds(lat, steps):
        t0 = time.perf_counter()
        lat.step(steps).synchronize()
        return time.perf_counter() - t0

    def lattice(nz):
        return lcbp.Lattice(dims[0], dims[1], nz, dtype=dtype).init_q(lcbp.BPII, 0.3).init_f_equilibrium(1.0)

    lattice(3).step(1).synchronize()  # the kernels' code is loaded
    first = []
    for k in range(3):  # a shape is tuned once in a process: others of about its size
        lat = lattice(dims[2] + k)
        lat.synchronize()
        first.append(seconds(lat, 1))
    seconds(lat, 64)
    assert min(first) < 700 * min(seconds(lat, 64) for _ in range(3)) / 64


@pytest.mark.parametrize("dims", [(64, 64, 255), (30, 61, 300), (126, 9, 601)])
def test_window_convolutions_of_many_plane_pairs(lcbp, dims):
    """Lattices that give a pipeline of the window kernel many plane pairs: the ring
    of accumulators and of staged planes wraps, ranges start inside a tile, a lone
    last plane.  Weights of -1, 0, 1 (two in a hundred not zero) and whole inputs keep every
    FP32 sum a whole number below 2^24, exact in any order, so the two kernels
    agree to the bit."""
    nx, ny, nz = dims
    rng = np.random.default_rng(12)
    q5 = rng.integers(-1, 2, size=(5, nz, ny, nx)).astype(np.float32)
    zero3, zero5 = np.zeros((3, nz, ny, nx), np.float32), np.zeros((5, nz, ny, nx), np.float32)
    out = []
    for kernel in (lcbp.CONV_TAPS, lcbp.CONV_WINDOW):
        sur = lcbp.Surrogate(nx, ny, nz)
        w = np.random.default_rng(13).choice([-1.0, 0.0, 1.0], p=[0.01, 0.98, 0.01], size=sur.get_params().size)
        sur.set_conv_kernel(kernel).set_params(w)
        out.append(sur.forward(q5, zero3, zero5, 2.0, -1.0))
        sur.close()
    assert np.abs(out[0]).max() > 0
    assert np.array_equal(out[0], out[1])


def test_loss_with_fractional_masks(lcbp):
    """The mask's weights sum on the device.  A constant 1/4 changes neither loss nor
    gradients (powers of two are exact), and loss times sum is additive in the mask:
    products rounded to FP32 (2^-24 each, three losses) and FP64 sums of positive terms."""
    shape = (6, 10, 33)
    rng = np.random.default_rng(3)
    q5, r5, dq = (0.1 * rng.standard_normal((5,) + shape) for _ in range(3))
    u3 = 1e-3 * rng.standard_normal((3,) + shape)
    m1 = rng.choice([0.0, 0.3, 0.7, 1.0], size=shape).astype(np.float32)
    m2 = (np.float32(1) - m1).astype(np.float32)
    sur = lcbp.Surrogate(shape[2], shape[1], shape[0], training=True)
    params = 0.02 * rng.standard_normal(sur.get_params().size)
    loss, grads = {}, {}
    for name, m in (("none", None), ("quarter", np.full(shape, 0.25, np.float32)), ("one", m1), ("rest", m2)):
        m64 = None if m is None else m.astype(np.float64)
        loss[name] = sur.set_params(params).train_step(q5, u3, r5, 1.0, -0.5, dq, m64, lr=1e-6)
        grads[name] = sur.get_grads()
    assert loss["quarter"] == loss["none"]
    assert np.array_equal(grads["quarter"], grads["none"])
    s1, s2 = m1.astype(np.float64).sum(), m2.astype(np.float64).sum()
    whole = loss["one"] * s1 + loss["rest"] * s2
    assert abs(whole - loss["none"] * m1.size) <= 4 * 2.0 ** -24 * loss["none"] * m1.size


def test_surrogate_reads_device_fields_in_place(lcbp):
    """CUDA float32 tensors, one value off a 16-byte boundary, give what the same numpy arrays give, to the bit."""
    import torch
    shape = (9, 10, 34)
    rng = np.random.default_rng(5)
    fields = [(0.1 * rng.standard_normal((c,) + shape)).astype(np.float32) for c in (5, 3, 5, 5)]
    mask = rng.choice([0.0, 0.5, 1.0], size=shape).astype(np.float32)

    def device(a):
        flat = torch.empty(a.size + 1, device="cuda")
        view = flat[1:].view(a.shape)
        view.copy_(torch.from_numpy(a))
        return view

    params = 0.02 * rng.standard_normal(lcbp.Surrogate(34, 10, 9).get_params().size)
    got = []
    for put in (lambda a: a, device):
        q, u, r, dq = (put(a) for a in fields)
        sur = lcbp.Surrogate(34, 10, 9, training=True).set_params(params)
        y = sur.forward(q, u, r, 1.0, -0.5)
        losses = [sur.train_step(q, u, r, 1.0, -0.5, dq, m, lr=1e-3) for m in (put(mask), None)]
        got.append((y, losses, sur.get_grads(), sur.get_params()))
        sur.close()
    assert got[0][1] == got[1][1]
    for k in (0, 2, 3):
        assert np.array_equal(got[0][k], got[1][k])


@pytest.mark.parametrize("dtype,mode", [("f32", "flow"), ("f32", "seidel"), ("f32", "noflow"), ("f64", "walls")])
def test_legacy_stream(lcbp, dtype, mode):
    """A lattice on the legacy stream (no capture, dependent launches one by one) steps as one on its own stream does,
    to the bit."""
    import ctypes
    import torch
    a = pair(lcbp, (10, 12, 36), dtype, mode)[0]
    b = pair(lcbp, (10, 12, 36), dtype, mode)[0]
    L = lcbp.lib()
    nbytes = L.lcbp_workspace_bytes(36, 12, 10, a.state_dtype)
    ws = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    handle = type(a._h)()
    lcbp.check(L.lcbp_create_on_buffers(36, 12, 10, a.state_dtype, ws.data_ptr() + (-ws.data_ptr()) % 256, nbytes, None,
                                        ctypes.byref(handle)))
    own = b._h, b._ws
    b._h, b._ws = handle, ws
    b.set_flow(flow_on="noflow" not in mode, coupling=lcbp.GAUSS_SEIDEL if "seidel" in mode else lcbp.JACOBI)
    if "walls" in mode:
        b.set_walls(True, (0.2, 0.0, 0.0, -0.1, 0.0))
    b.set_q(a.read_q())
    if "noflow" not in mode:
        b.set_f(a.read_f())
        a.set_f(a.read_f())
    for lat in (a, b):
        lat.step(51).step(1)
    assert np.array_equal(a.read_q(), b.read_q())
    if "noflow" not in mode:
        assert np.array_equal(a.read_f(), b.read_f())
    b.close()
    b._h, b._ws = own
