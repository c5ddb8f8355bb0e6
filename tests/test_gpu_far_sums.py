"""The far-field sums and their adjoint on inputs at the edge of what the tap tables hold.

* Directions longer than a unit vector (r.r' / c counts as the delay whatever the length)
  span more steps than an RWG does along a unit vector: against the plain evaluation of
  test_gpu_fields, with its tolerance.
* A value does not depend on the other directions and times of the call (bitwise), also where
  the call takes several passes over either.
* The work space of a larger call takes the place of a smaller call's, and a march with the
  far field allocates nothing after its first step.
* An infinite or undefined current (or adjoint input) reaches the times that its support
  touches and no others, which are those of a call without it, bitwise.
* More steps than a grid dimension holds tiles for: the last steps equal those of a short call
  with the times moved along, and the far field of the first ones that of a short call.
"""
import math

import numpy as np
import pytest

from paper_1408_7060_gb300.inputs import random_plane_waves
from test_gpu_fields import C0, MU0, context, d_basis, surface

pytestmark = pytest.mark.gpu


def plain(c, V, F, order, dt, f_c, dirs, I, n0, G_in):
    """Far field of I [steps][ns] at n0 .. and the adjoint of G_in [n_out][nd][2]."""
    rh, e1, e2 = dirs
    r, wS = surface(c, V, F)
    wc = 2 * math.pi * f_c
    out, adj = np.zeros_like(G_in), np.zeros_like(I)
    for d in range(len(rh)):
        rr = r @ rh[d]
        ph = -MU0 / (4 * math.pi) * np.exp(1j * wc / C0 * rr)
        taps = {}
        for i in range(len(G_in)):
            for l in range(len(I)):
                s = n0 + i - (l + 1)
                if s not in taps:
                    t = d_basis(s + rr / (C0 * dt), order, dt, wc) * ph
                    taps[s] = np.stack([(t * (wS @ e1[d])).sum(1), (t * (wS @ e2[d])).sum(1)], 1)
                out[i, d] += I[l] @ taps[s]
                adj[l] += taps[s].conj() @ G_in[i, d]
    return out, adj


@pytest.mark.parametrize("order,cdt,length", [(2, 0.8, 1.7), (1, 0.8, 3.0), (3, 0.8, 10.0), (2, 0.8, 0.3)])
def test_directions_of_any_length(order, cdt, length):
    from paper_1408_7060_gb300 import abi

    f_c, dt, n0, steps, n_out, nd = 150e6, cdt / C0, -12, 9, 40, 5
    V, F, c = context(1, order, dt, f_c)
    with c:
        rh, e1 = random_plane_waves(nd, 2)
        e2 = np.cross(rh, e1)
        rh = rh * np.array([1.0, length, 1.0, length, 0.5])[:, None]
        rng = np.random.default_rng(5)
        I = rng.standard_normal((steps, c.ns)) + 1j * rng.standard_normal((steps, c.ns))
        G_in = rng.standard_normal((n_out, nd, 2)) + 1j * rng.standard_normal((n_out, nd, 2))
        ref, radj = plain(c, V, F, order, dt, f_c, (rh, e1, e2), I, n0, G_in)
        got = abi.aim_farfield(c.handle, rh, e1, e2, I, n0, n_out)
        adj = abi.aim_farfield_adjoint(c.handle, rh, e1, e2, steps, n0, G_in)
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
    assert np.abs(adj - radj).max() <= 1e-12 * np.abs(radj).max()


@pytest.mark.parametrize("sub,nd,n_out", [(2, 40, 150), (3, 9, 300), (1, 2600, 130), (3, 600, 70)])
def test_a_value_alone_and_among_others(sub, nd, n_out):
    from paper_1408_7060_gb300 import abi

    f_c, dt, n0, steps = 150e6, 0.5 / C0, -6, 40
    V, F, c = context(sub, 2, dt, f_c)
    with c:
        rh, e1 = random_plane_waves(nd, 2)
        e2 = np.cross(rh, e1)
        rng = np.random.default_rng(5)
        I = rng.standard_normal((steps, c.ns)) + 1j * rng.standard_normal((steps, c.ns))
        got = abi.aim_farfield(c.handle, rh, e1, e2, I, n0, n_out)
        for d, i, k in ((0, 0, 20), (nd - 1, 3, 40), (nd // 2, 11, 1)):
            one = slice(d, d + 1)
            alone = abi.aim_farfield(c.handle, rh[one], e1[one], e2[one], I, n0 + i, k)
            assert np.array_equal(alone[:, 0], got[i:i + k, d]), (d, i, k)


def device_bytes(c):
    from paper_1408_7060_gb300 import abi

    return abi.aim_get_info(c.handle)["device_bytes"]


def test_work_space_is_not_left_behind():
    from paper_1408_7060_gb300 import abi

    held = []
    for sizes in ((20, 30, 45, 70, 100), (100,)):
        V, F, c = context(2, 2, 0.5 / C0, 150e6)
        with c:
            rh, e1 = random_plane_waves(12, 2)
            e2 = np.cross(rh, e1)
            for n in sizes:
                abi.aim_farfield(c.handle, rh, e1, e2, np.ones((n, c.ns), complex), -3, n + 6)
            held.append(device_bytes(c))
    assert held[0] == held[1]


def test_a_march_allocates_before_its_first_step():
    from paper_1408_7060_gb300 import abi

    k, p = random_plane_waves(1, 1)
    a = np.ones(6, complex)
    held = []
    for steps in (1, 12):
        V, F, c = context(2, 2, 0.5 / C0, 150e6)
        with c:
            rh, e1 = random_plane_waves(12, 2)
            abi.aim_march_farfield(c.handle, k[0], p[0], 0, a, steps, 1e-3, rh, e1, np.cross(rh, e1), 0, 40)
            held.append(device_bytes(c))
    assert held[0] == held[1]


@pytest.mark.parametrize("bad", [np.inf, np.nan])
@pytest.mark.parametrize("order,cdt", [(1, 0.9), (2, 0.6), (4, 1.2)])
def test_non_finite_values_stay_within_their_support(order, cdt, bad):
    from paper_1408_7060_gb300 import abi

    f_c, dt, n0, steps, n_out, nd = 150e6, cdt / C0, -8, 20, 40, 9
    V, F, c = context(2, order, dt, f_c)
    with c:
        r, _ = surface(c, V, F)
        rh, e1 = random_plane_waves(nd, 2)
        e2 = np.cross(rh, e1)
        rng = np.random.default_rng(5)
        I = rng.standard_normal((steps, c.ns)) + 1j * rng.standard_normal((steps, c.ns))
        G = rng.standard_normal((n_out, nd, 2)) + 1j * rng.standard_normal((n_out, nd, 2))
        far = abi.aim_farfield(c.handle, rh, e1, e2, I, n0, n_out)
        adj = abi.aim_farfield_adjoint(c.handle, rh, e1, e2, steps, n0, G)
        k, j = 77, 9                                           # the RWG and the step (from 0)
        I[j, k] = bad
        got = abi.aim_farfield(c.handle, rh, e1, e2, I, n0, n_out)
        i, d = 21, 4
        G[i, d, 1] = bad
        gadj = abi.aim_farfield_adjoint(c.handle, rh, e1, e2, steps, n0, G)
    w = r @ rh.T / (C0 * dt)                                   # [ns][14][nd]
    inside = lambda u: (u > -1) & (u <= order)
    n = n0 + np.arange(n_out)
    reach = inside((n - (j + 1))[:, None, None] + w[k][None]).any(1)          # [n_out][nd]
    assert np.array_equal(got[~reach], far[~reach]) and not np.isfinite(got[reach]).all(-1).any()
    l = 1 + np.arange(steps)
    reach = inside((n0 + i - l)[:, None, None] + w[None, :, :, d]).any(-1)    # [steps][ns]
    assert np.array_equal(gadj[~reach], adj[~reach]) and not np.isfinite(gadj[reach]).any()


def test_more_steps_than_a_grid_dimension():
    import torch

    from paper_1408_7060_gb300 import AimContext, abi
    from paper_1408_7060_gb300.inputs import place_grid, plate_mesh

    V, F = plate_mesh(0.3, 2)
    h, origin = place_grid(V, 16)
    steps, tail, nd, n_out = 65535 * 64 + 200, 50, 3, 9
    with AimContext(V=V, F=F, grid_n=16, origin=origin, h=h, near_radius=-1.0, dt=0.5 / C0, f_c=150e6,
                    precision="c128") as c:
        rh, e1 = random_plane_waves(nd, 2)
        e2 = np.cross(rh, e1)
        G = torch.randn(n_out, nd, 2, dtype=torch.complex128, device="cuda")
        long = abi.aim_farfield_adjoint(c.handle, rh, e1, e2, steps, steps - 5, G)
        short = abi.aim_farfield_adjoint(c.handle, rh, e1, e2, tail, tail - 5, G)
        assert torch.equal(long[-tail:], short) and float(short.abs().max()) > 0
        far = abi.aim_farfield(c.handle, rh, e1, e2, long, steps - 40, steps + 30)
        assert torch.equal(far[:60], abi.aim_farfield(c.handle, rh, e1, e2, long[-90:].contiguous(), 50, 60))
        assert float(far[60:].abs().max()) == 0.0
