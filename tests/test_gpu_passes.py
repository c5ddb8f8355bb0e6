"""Passes that few set-ups reach, every right-hand side of a batch, and what a batch may not
change.  The path (plane kernel, or separate y and z passes) is read from the launch counts.

* The separate passes on z-spectra (power-of-two z lengths whose plane does not fit shared
  memory): products and delayed sums against the plain evaluation of test_gpu_plane, and the
  blocked march against the direct one within the solves' tolerance, so that the elementwise
  square, the pending inverse and both kernels of the streamed delay sum run.  The bounds are
  those of test_gpu_blocked; the complex64 one holds for RWGs of two or three grid spacings (the
  30 720-RWG sphere on 128^3: 2.4e-6), while on coarser meshes the grid part is far larger than
  the product it is a part of and both marches are equally far from the complex128 one (7680
  RWGs: 3.9e-5 each, and 2.2e-5 from one another).
* Remaining pairs of padded and z lengths of the plane kernel, every right-hand side.
* A product, a delayed sum and a march of several right-hand sides are bitwise those of each
  alone (products and sums) or those to 1e-10 (marches: the bound of the batched sphere), on the
  plane kernel with the paired gather, and on the 384^3 grid, where a warp runs through all
  right-hand sides of its columns and leaves out those that have converged.
"""
import numpy as np
import pytest

from paper_1408_7060_gb300.inputs import icosphere, place_grid, random_plane_waves, sphere_array
from test_gpu_plane import BAND, F_C, Plain, geometry

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(np.ravel(a - b)) / np.linalg.norm(np.ravel(b))


def launches(c, kind):
    return c.get_profile()[0][kind][0]


def crandn(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


# (mesh, size, grid, z length, precision, right-hand sides, separate passes)
SIZES = [("sphere2", 0.12, 96, 32, "c64", 3, False), ("sphere2", 0.12, 96, 32, "c128", 2, False),
         ("sphere2", 0.25, 96, 64, "c64", 3, False), ("sphere2", 0.25, 96, 64, "c128", 2, True),
         ("sphere2", 0.09, 128, 32, "c64", 3, False), ("sphere2", 0.09, 128, 32, "c128", 2, True),
         ("sphere2", 0.2, 128, 64, "c64", 3, False), ("sphere2", 0.2, 128, 64, "c128", 2, True),
         ("sphere2", 1.0, 64, 128, "c128", 2, True), ("sphere2", 0.4, 64, 64, "c128", 2, True),
         ("sphere2", 0.15, 64, 32, "c128", 2, False), ("sphere2", 1.0, 32, 64, "c128", 2, False),
         ("sphere2", 0.5, 96, 128, "c128", 2, True), ("sphere2", 0.4, 128, 128, "c128", 2, True),
         ("sphere2", 0.53, 128, 144, "c128", 1, True), ("sphere2", 0.7, 128, 192, "c64", 3, True),
         ("sphere2", 1.0, 128, 256, "c64", 2, True), ("plate", 14, 384, 16, "c64", 2, True)]


@pytest.mark.parametrize("mesh,size,grid,lz,precision,nb,separate", SIZES)
def test_every_right_hand_side(mesh, size, grid, lz, precision, nb, separate):
    from paper_1408_7060_gb300 import AimContext

    V, F, h, origin = geometry(mesh, size, grid)
    rng = np.random.default_rng(3)
    eps = 2.0 ** -53 if precision == "c128" else 2.0 ** -24
    with AimContext(V=V, F=F, grid_n=grid, origin=origin, h=h, near_radius=3 * h, dt=0.25 / (BAND * F_C), f_c=F_C,
                    precision=precision, batch_max=nb) as c:
        assert c.info["z_len"] == lz
        plain = Plain(c)
        x, hist = crandn(rng, nb, c.ns), crandn(rng, c.n_delays, nb, c.ns)
        got, sums = c.matvec(0, x), c.rhs(2, hist)            # step 2: the delay 1 alone
        assert (launches(c, "yfft_fwd") > 0) == separate
        for b in range(nb):
            for y, (ref, scale) in ((got[b], plain.product(0, x[b])), (sums[b], plain.product(1, hist[0, b]))):
                assert np.linalg.norm(y - ref) < 8 * eps * scale, b


@pytest.mark.parametrize("sub,grid,z,lz,precision,tol,bound", [(5, 128, 1.0, 256, "c64", 1e-6, 1e-5),
                                                              (4, 96, 0.5, 128, "c128", 1e-10, 1e-9)])
def test_blocked_march_on_the_separate_passes(sub, grid, z, lz, precision, tol, bound):
    from paper_1408_7060_gb300 import AimContext

    V, F = icosphere(sub, 1.0)
    V = V * np.array([1.0, 1.0, z])
    h, origin = place_grid(V, grid)
    f_c, band = 600e6, 0.3
    k, p = random_plane_waves(1, 1)
    sigma = 3 / (2 * np.pi * band * f_c)
    got = []
    for blocked in (0, 1):
        with AimContext(V=V, F=F, grid_n=grid, origin=origin, h=h, near_radius=0.1 if sub == 5 else 0.15,
                        dt=0.25 / (band * f_c), f_c=f_c, precision=precision, precond="sai",
                        precond_radius=0.08 if sub == 5 else 0.15, rhs_blocked=blocked) as c:
            assert c.info["z_len"] == lz and c.n_delays > 4
            got.append(c.march(k, p, sigma, 4 * sigma, 12, tol)[0])
            assert launches(c, "yfft_fwd") > 0
            assert (launches(c, "block_square") > 0) == (launches(c, "zinv_pending") > 0) == bool(blocked)
    assert rel(got[1], got[0]) < bound


@pytest.mark.parametrize("batch_max", [5, 6])
def test_batch_is_bitwise_its_vectors_on_the_plane_kernel(batch_max):
    from paper_1408_7060_gb300 import AimContext

    V, F = icosphere(4, 1.0)
    h, origin = place_grid(V, 64)
    rng = np.random.default_rng(6)
    with AimContext(V=V, F=F, grid_n=64, origin=origin, h=h, near_radius=3 * h, dt=0.25 / 180e6, f_c=600e6,
                    precision="c64", batch_max=batch_max) as c:
        x, hist = crandn(rng, 5, c.ns), crandn(rng, c.n_delays, 5, c.ns)
        got, sums = c.matvec(1, x), c.rhs(c.n_delays + 1, hist)
        for b in range(5):
            assert np.array_equal(c.matvec(1, x[b:b + 1])[0], got[b]), b
            assert np.array_equal(c.rhs(c.n_delays + 1, np.ascontiguousarray(hist[:, b:b + 1]))[0], sums[b]), b


def test_batch_is_its_vectors_on_the_largest_grid():
    from paper_1408_7060_gb300 import AimContext, abi

    V, F = sphere_array(4, 0.5, 1.5)
    h, origin = place_grid(V, 384)
    rng = np.random.default_rng(6)
    with AimContext(V=V, F=F, grid_n=384, origin=origin, h=h, near_radius=3 * h, dt=0.25 / 50e6, f_c=1e9,
                    precision="c64", batch_max=3, precond="sai", precond_radius=4.2 * h) as c:
        assert c.info["z_len"] == 144
        x = crandn(rng, 3, c.ns)
        got = c.matvec(0, x)
        for b in range(3):
            assert np.array_equal(c.matvec(0, x[b:b + 1])[0], got[b]), b
        # the waves of a solve converge at different iterations (the one without a source at none)
        src = crandn(rng, 2, 3, c.ns)
        src[:, 1] = 0.0
        src[:, 2] = c.matvec(0, x[:1] / np.abs(x[:1]))[0]
        cur, st, _ = abi.aim_march_source(c.handle, src, 1e-2)
        assert (st["iters"][0, 1] == 0) and (st["iters"][0, [0, 2]] > 0).all() and np.all(cur[:, 1] == 0)
        for b in (0, 2):
            one, so, _ = abi.aim_march_source(c.handle, np.ascontiguousarray(src[:, b:b + 1]), 1e-2)
            assert rel(cur[:, b], one[:, 0]) < 1e-10 and np.array_equal(st["iters"][:, b], so["iters"][:, 0])


@pytest.mark.parametrize("precision,tol,bound", [("c128", 1e-10, 1e-9), ("c64", 1e-6, 1e-5)])
def test_blocked_march_of_several_waves_on_the_plane_kernel(precision, tol, bound):
    """Blocked and direct marches of three waves of a context for four (bounds of test_gpu_blocked)."""
    from paper_1408_7060_gb300 import AimContext
    from paper_1408_7060_gb300.inputs import make_workload

    w = make_workload("sphere480", band_frac=0.2, n_t=24)
    k, p = random_plane_waves(3, 5)
    got = []
    for blocked in (0, 1):
        with AimContext.from_workload(w, precision=precision, batch_max=4, rhs_blocked=blocked) as c:
            got.append(c.march(k, p, w.sigma, w.t_d, w.n_t, tol)[0])
            assert launches(c, "yfft_fwd") == 0 and (launches(c, "block_square") > 0) == bool(blocked)
    assert all(rel(got[1][:, b], got[0][:, b]) < bound for b in range(3))
