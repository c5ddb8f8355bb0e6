"""What a set-up does when device memory is short: most of the device is held by another
allocation while a context of a factor-3 z length (96^3, a ring of several GB) is made.

* Where the context fits, it runs the kernels that it would run on an empty device, with
  bitwise the same results: the choice between the plane kernel and the separate y and z
  passes follows from the sizes alone.
* Where the plane path's ring does not fit but that of the separate passes does, the set-up
  goes through with the separate passes: buffers, launch plan and warm-up of that path, none
  of the other's memory kept, products and marches within the complex64 rounding of the grid.

A context of the plane kernel holds no slab of the separate passes, in either precision.
"""
import contextlib

import numpy as np
import pytest

from paper_1408_7060_gb300.inputs import icosphere, place_grid, random_plane_waves

pytestmark = pytest.mark.gpu

F_C, BAND, GB = 600e6, 0.3, 1 << 30


@contextlib.contextmanager
def only(free_bytes):
    """Leave about free_bytes of device memory free."""
    import torch

    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    held = torch.empty(free - free_bytes, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del held
        torch.cuda.empty_cache()


def context(**kw):
    from paper_1408_7060_gb300 import AimContext

    V, F = icosphere(4, 1.0)
    h, origin = place_grid(V, 96)
    return AimContext(V=V, F=F, grid_n=96, origin=origin, h=h, near_radius=0.15, dt=0.25 / (BAND * F_C), f_c=F_C,
                      precision="c64", batch_max=8, precond="sai", precond_radius=0.25, **kw)


def passes(c, x, hist):
    """Product, delayed sum, a short march, and whether the separate y passes ran."""
    y, r = c.matvec(0, x), c.rhs(c.n_delays + 1, hist)
    k, p = random_plane_waves(2, 1)
    sigma = 3 / (2 * np.pi * BAND * F_C)
    cur, _, _ = c.march(k, p, sigma, 4 * sigma, 4, 1e-5)
    return (y, r, cur), c.get_profile()[0]["yfft_fwd"][0] > 0


def inputs(c):
    rng = np.random.default_rng(4)
    x = rng.standard_normal((8, c.ns)) + 1j * rng.standard_normal((8, c.ns))
    hist = rng.standard_normal((c.n_delays, 8, c.ns)) + 1j * rng.standard_normal((c.n_delays, 8, c.ns))
    return x, hist


def rel(a, b):
    return np.linalg.norm(np.ravel(a - b)) / np.linalg.norm(np.ravel(b))


def test_path_follows_from_the_sizes(tmp_path, monkeypatch):
    from paper_1408_7060_gb300 import abi

    monkeypatch.setenv("AIM_GB300_PLAN_CACHE", str(tmp_path / "plans.jsonl"))
    with context() as c:
        assert c.info["z_len"] == 192
        data, full = inputs(c), c.info["device_bytes"]
        ring = c.n_delays * 8 * 4 * 192 ** 3 * 8
        want, separate = passes(c, *data)
    assert not separate and ring > 4 * GB
    with only(full + 6 * GB):
        assert ring > (full + 6 * GB) // 4
        with context() as c:
            got, separate = passes(c, *data)
            assert not separate
    assert all(np.array_equal(a, b) for a, b in zip(got, want))
    # a quarter of the ring short: the separate passes
    with only(full - ring // 4):
        with context(autotune=2) as c:
            got, separate = passes(c, *data)
            assert separate and c.info["device_bytes"] < full - ring // 3
            assert c.info["plan_source"] == abi.AIM_PLAN_MEASURED
    assert all(rel(a, b) < 1e-5 for a, b in zip(got[:2], want[:2])) and rel(got[2], want[2]) < 1e-4


def plane_table(n, lz):
    """Bytes of the FP64 spectra of one delay in the plane kernel's order, at most."""
    return 2 * (n + 1) * 2 * n * lz * 16


@pytest.mark.parametrize("grid,precision", [(64, "c64"), (32, "c128")])
def test_no_slab_beside_the_plane_kernel(grid, precision):
    from paper_1408_7060_gb300 import AimContext

    V, F = icosphere(4, 1.0)
    h, origin = place_grid(V, grid)
    es = 8 if precision == "c64" else 16

    def held(**kw):
        kw = {"precision": precision, **kw}
        with AimContext(V=V, F=F, grid_n=grid, origin=origin, h=h, near_radius=3 * h, dt=0.25 / (BAND * F_C), f_c=F_C,
                        **kw) as c:
            assert c.info["z_len"] == 2 * grid
            c.matvec(0, np.ones((1, c.ns), complex))
            assert c.get_profile()[0]["yfft_fwd"][0] == 0
            nz, L = c.info["box_hi"][2] - c.info["box_lo"][2] + 1, 2 * grid
            # elements per wave: ring, A and P, slab
            return c.info["device_bytes"], c.n_delays * 4 * L ** 3, 4 * nz * grid * (L + grid), 4 * nz * L ** 2, c.ns

    # what 100 more waves take beyond their ring, A, P and vectors is less than their slab
    (b1, ring, work, slab, ns), more = held(), held(batch_max=101)[0]
    vectors = 100 * ns * 16 * (51 + 40)                        # Krylov basis, histories, work vectors
    assert more - b1 < 100 * (es * (ring + work) + es * slab // 2) + vectors
    if grid == 32:                                             # and the refinement's FP64 buffers likewise
        b1, more = held(precision="c64")[0], held(precision="c64", refine=2)[0]
        assert more - b1 < 16 * work + 16 * slab // 2 + plane_table(grid, 2 * grid)
