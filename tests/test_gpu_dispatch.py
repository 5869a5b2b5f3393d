"""Kernel dispatch and work distribution at the sizes where they can go wrong:
default tiles on both sides of the lines of the rule that picks them, blocks
that work through many tiles (more than the FD stage kernel has tile buffers
and descriptor slots), groups with more lattices than its lookup table holds,
and recorded observables of lattices with fewer, exactly as many and more
blocks than one block adds up.
"""
import numpy as np
import pytest

import lbm_workloads as wl
import oracle
import paper_1904_02471_gb300 as pkg
from paper_1904_02471_gb300 import lbm

pytestmark = pytest.mark.gpu

TOL64 = 1e-12   # populations after a few steps, as for the oracle parity tests
TAU = 0.8 / 3 ** 0.5
VMAX = {3: 3 ** 0.5, 4: 2.33441421833897723932, 5: 2.85697001387280565416}


@pytest.fixture(scope="module", autouse=True)
def gpu():
    import torch
    assert torch.cuda.is_available()
    from paper_1904_02471_gb300 import build
    build.build()
    torch.cuda.init()


def rel_err(a, b):
    return float(np.max(np.abs(a - b) / np.abs(b)))


def _state(q, nx, ny, seed):
    f = oracle.equilibrium(q, *wl.random_smooth(nx, ny, seed))
    return f * (1 + wl.random_uniform(f.shape, seed + 1, -0.02, 0.02))


def _fd(q, nx, ny, scheme, prec):
    dt = 0.3 / nx / VMAX[q]
    return pkg.Lattice("fd", q, nx, ny, dt / 5 if scheme == "imex" else 2 * dt, dt=dt, precision=prec, scheme=scheme)


@pytest.mark.parametrize("nx,ny", [(64, 4), (33, 3), (139, 139), (140, 140), (255, 257), (256, 256)])
def test_cs_default_tile_fp64(nx, ny):
    """19,456 and 65,536 nodes are the lines between the FP64 default tiles."""
    f0 = _state(3, nx, ny, 5)
    with pkg.Lattice("cs", 3, nx, ny, TAU) as L:
        L.set_populations(f0)
        L.step(5)
        assert rel_err(L.populations(), oracle.cs_run(f0, TAU, 5)) < TOL64


@pytest.mark.parametrize("storage", ["ab", "inplace"])
@pytest.mark.parametrize("nx", [2896, 2897])
def test_cs_default_tile_fp32_at_the_bulk_line(nx, storage):
    """8 Mi nodes: the plain kernel below, the bulk-copy kernel from there on;
    both are bit-identical to the other kernel's result."""
    ny = 2896
    rho, ux, uy = wl.taylor_green(nx, ny, 0.01)
    res = []
    for tile in (None, 0, 5):
        with pkg.Lattice("cs", 3, nx, ny, TAU, precision="fp32", storage=storage) as L:
            if tile is not None:
                L.config(tile)
            L.init(rho, ux, uy)
            L.step(3)
            res.append([L.populations_region(x0, y0, 40, 40) for x0, y0 in ((0, 0), (nx - 20, ny - 20), (1000, 2000))])
    for r in res[1:]:
        for a, b in zip(res[0], r):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("scheme", ["rk3", "imex"])
@pytest.mark.parametrize("q,nx,ny", [(4, 160, 96), (4, 31, 17), (3, 97, 33), (5, 66, 35), (4, 2048, 4)])
def test_fd_tiles_in_turn(q, nx, ny, scheme):
    """One block for all tiles, three, and the default: the same bits; FP64
    equal to the oracle."""
    f0 = _state(q, nx, ny, 9)
    res = []
    for tile, grid in ((None, 0), (0, 1), (0, 3), (1, 2), (2, 1), (3, 5)):
        with _fd(q, nx, ny, scheme, "fp32") as L:
            if tile is not None:
                L.config(tile, grid)
            L.set_populations(f0)
            L.step(4)
            res.append(L.populations())
    for r in res[1:]:
        assert np.array_equal(res[0], r)
    if nx * ny <= 4096:
        with _fd(q, nx, ny, scheme, "fp64") as L:
            s = L.spec
            L.config(3, 2)
            L.set_populations(f0)
            L.step(4)
            run = oracle.fd_imex_run if scheme == "imex" else oracle.fd_run
            assert rel_err(L.populations(), run(f0, s.dx, s.dt, s.tau, 4)) < TOL64


def test_more_lattices_than_the_lookup_table():
    """260 lattices in one FD group, some with a spent budget: each advances
    as it does alone."""
    n, dt = 12, 0.3 / 12 / VMAX[4]
    specs = [pkg.make_spec("fd", 4, n, n + i % 3, 2 * dt, dt, 0.0, "fp64") for i in range(260)]
    f = {}
    B = pkg.Batch(specs)
    try:
        for i, s in enumerate(specs):
            B.init(i, *wl.random_smooth(s.nx, s.ny, 100 + i % 7))
            if i % 5 == 0:
                B.set_budget(i, 2)
        B.step(4)
        for i in (0, 1, 5, 128, 255, 256, 259):
            f[i] = B.populations(i)
    finally:
        B.close()
    for i, got in f.items():
        s = specs[i]
        ref = oracle.fd_run(oracle.equilibrium(4, *wl.random_smooth(s.nx, s.ny, 100 + i % 7)), 1 / s.nx, dt, 2 * dt,
                            2 if i % 5 == 0 else 4)
        assert rel_err(got, ref) < TOL64, i


# blocks of a launch: 255, 256, 257, 520 (one block adds up 256 of them), 5200
# (finished by a launch of its own), and FD stages, whose blocks do several tiles
@pytest.mark.parametrize("model,q,nx,ny,tile,scheme", [
    ("cs", 3, 32, 255, 7, "rk3"), ("cs", 3, 32, 256, 7, "rk3"), ("cs", 3, 31, 257, 7, "rk3"), ("cs", 3, 97, 130, 7, "rk3"),
    ("cs", 3, 300, 520, 7, "rk3"), ("cs", 3, 1030, 70, 6, "rk3"), ("fd", 4, 64, 256, 3, "rk3"), ("fd", 4, 200, 90, 3, "rk3"),
    ("fd", 5, 66, 171, 3, "imex"), ("fd", 4, 200, 157, 1, "rk3_fused")])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_recorded_sums_equal_the_snapshot(model, q, nx, ny, tile, scheme, prec):
    """The record written by the last block of a step against the sums of the
    state read out on its own, at the same step. FP32 kernels add up to 32
    lanes' float sums of a few nodes in float: each addition rounds by 2^-24 of
    the magnitudes summed so far, at most 40 of them per node's path."""
    rho, ux, uy = wl.random_smooth(nx, ny, 3, amp_u=0.02)
    px, py = np.sin(2 * np.pi * np.arange(nx) / nx), np.cos(2 * np.pi * np.arange(ny) / ny)
    if model == "cs":
        L = pkg.Lattice("cs", 3, nx, ny, TAU, precision=prec)
    else:
        L = _fd(q, nx, ny, scheme, prec)
    with L:
        L.config(tile)
        L.init(rho, ux, uy)
        L.set_probe(0, px, py, 1.0)
        L.record(3, 10)
        snaps = []
        for _ in range(3):
            o, (r, u, v) = L.observables(), L.moments()
            w = np.abs(u * px[None, :] * py[:, None]).sum()
            snaps.append((o, np.abs(r - 1).sum(), np.abs(r * u).sum(), np.abs(r * v).sum(), w))
            L.step(3)
        L.sync()
        ser = L.series()
    eps = 2.0 ** -53 * nx * ny if prec == "fp64" else 40 * 2.0 ** -24
    assert [s["step"] for s in ser] == [0, 3, 6]
    for s, (o, mr, mu, mv, mw) in zip(ser, snaps):
        full = nx * ny if prec == "fp64" else mr   # FP64 stores f itself, FP32 deviations
        assert abs(s["mass"] - o["mass"]) <= eps * full + 1e-12
        assert abs(s["mom_x"] - o["mom_x"]) <= eps * max(mu, full) and abs(s["mom_y"] - o["mom_y"]) <= eps * max(mv, full)
        assert abs(s["amp"] - o["amp"]) <= eps * max(mw, 1e-3 * full)
        assert s["nonfinite"] == 0


@pytest.mark.parametrize("scheme", ["rk3", "imex", "rk3_fused"])
@pytest.mark.parametrize("q", [3, 4, 5])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_fd_equilibrium_of_negative_density(q, scheme, prec):
    """Eq. (herfeq) is odd in f: -f is a state like f, and its run is the run of
    f with the sign changed. FP32 stores float32(f - w rho0), here of size
    2 w: one rounding of 2^-24 of that per stage (12 of them) and in each
    equilibrium and flux, amplified by less than 10 over four steps."""
    nx, ny = 45, 22
    f0 = _state(q, nx, ny, 13)
    with _fd(q, nx, ny, scheme, prec) as L:
        s = L.spec
        L.set_populations(-f0)
        L.step(4)
        got = L.populations()
    run = oracle.fd_imex_run if scheme == "imex" else oracle.fd_run
    ref = run(-f0, s.dx, s.dt, s.tau, 4)
    assert rel_err(got, ref) < (TOL64 if prec == "fp64" else 12 * 2 * 10 * 2.0 ** -24)


@pytest.mark.parametrize("prec,scheme", [("fp32", "rk3"), ("fp32", "imex"), ("fp64", "rk3")])
@pytest.mark.parametrize("nx", [7, 29, 30, 31, 33, 34, 35, 61, 63, 65, 66, 99])
def test_fd_ragged_width(nx, prec, scheme):
    """Widths around a tile's edge with every remainder of a 16-byte copy: the
    copies across the periodic edge and the ones left out beyond it. FP32
    tolerance as above."""
    f0 = _state(4, nx, 19, 17)
    with _fd(4, nx, 19, scheme, prec) as L:
        s = L.spec
        L.set_populations(f0)
        L.step(4)
        got = L.populations()
    run = oracle.fd_imex_run if scheme == "imex" else oracle.fd_run
    assert rel_err(got, run(f0, s.dx, s.dt, s.tau, 4)) < (TOL64 if prec == "fp64" else 12 * 2 * 10 * 2.0 ** -24)
