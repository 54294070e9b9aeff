"""The kernels that AUTO picks for each kind of step against the generic ones.

Widths that are no multiple of 4 (the z-marching kernels with plain row
prefetches), steps with the flow off (the Heun kernels on the Q mirror) and
Gauss-Seidel coupling (the LB halves of the z-marching kernels, then the Heun
kernels with the new velocity), with and without walls, on shapes with ragged tiles in x and y, several tiles and
z-chunks, and the smallest width.
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


# 128 positions per CTA: one partly filled CTA, several, a width of 32 lanes; the
# longest chunk (16 planes) with a shorter last one
@pytest.mark.parametrize("mode", ["noflow", "noflow_walls"])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shape", [(3, 5, 4), (1, 11, 13), (37, 19, 45), (8, 16, 32), (50, 160, 250)])
def test_heun_kernels_match_generic(lcbp, shape, dtype, mode):
    check(lcbp, shape, dtype, mode, 10)


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
