"""Far-field envelopes, their adjoint and the RCS against a plain numpy evaluation of the
same cubature, at the sizes where the kernels' tiles end: one and several tiles of
directions, times and RWGs, right-hand sides beyond one pass, time steps so short that an
RWG spans more steps than the tap tables hold, faces so large that the phases inside one
exceed the series' range.

Tolerance 1e-12 of the largest result (FP64 sums of a few thousand terms of both signs;
the time derivative of the basis adds a factor of about 10).
"""
import math

import numpy as np
import pytest

from paper_1408_7060_gb300.inputs import icosphere, place_grid, random_plane_waves

pytestmark = pytest.mark.gpu

C0, MU0 = 299792458.0, 4e-7 * math.pi


def context(sub, order, dt, f_c):
    from paper_1408_7060_gb300 import AimContext

    V, F = icosphere(sub, 1.0)
    h, origin = place_grid(V, 16, 0.15)
    return V, F, AimContext(V=V, F=F, grid_n=16, origin=origin, h=h, near_radius=-1.0, dt=dt, f_c=f_c, order=order,
                            precision="c128")


def surface(c, V, F):
    """Cubature points [ns][14][3] and weighted basis functions of every RWG."""
    s15 = math.sqrt(15.0)
    b, w = [(1 / 3, 1 / 3, 1 / 3)], [9 / 40]
    for sg in (-1.0, 1.0):
        p = (6.0 + sg * s15) / 21.0
        for i in range(3):
            q = [p, p, p]
            q[i] = 1.0 - 2.0 * p
            b.append(tuple(q))
            w.append((155.0 + sg * s15) / 1200.0)
    edge, tri, free = c.rwg_table()
    T = V[F]
    area = 0.5 * np.linalg.norm(np.cross(T[:, 1] - T[:, 0], T[:, 2] - T[:, 0]), axis=1)
    ln = np.linalg.norm(V[edge[:, 0]] - V[edge[:, 1]], axis=1)
    r = np.einsum("qv,kavd->kaqd", np.array(b), T[tri])
    S = (np.array([1.0, -1.0]) * ln[:, None] / (2.0 * area[tri]))[:, :, None, None] * (r - V[free][:, :, None, :])
    wt = np.array(w)[None, None, :] * area[tri][:, :, None]
    return r.reshape(c.ns, 14, 3), (wt[..., None] * S).reshape(c.ns, 14, 3)


def d_basis(u, Q, dt, wc):
    T, D = np.zeros_like(u), np.zeros_like(u)
    for j in range(Q + 1):
        on = (u > j - 1) & (u <= j)
        t, d = np.ones_like(u), np.zeros_like(u)
        for i in range(j - Q, j + 1):
            if i != 0:
                d = d * (u - i) / (-i) + t / (-i)
                t = t * (u - i) / (-i)
        T, D = np.where(on, t, T), np.where(on, d, D)
    return D / dt + 1j * wc * T


# (subdivision, order, c dt in m, directions, steps, far times): the last two hold several
# steps per RWG, one within the tap tables and one beyond them
@pytest.mark.parametrize("sub,order,cdt,nd,steps,n_out", [(1, 2, 0.8, 1, 1, 3), (1, 3, 0.8, 5, 9, 70),
                                                         (2, 1, 0.5, 17, 66, 20), (2, 4, 1.0, 4, 5, 64),
                                                         (1, 2, 0.3, 6, 20, 40), (1, 3, 0.1, 3, 30, 50)])
def test_far_field_and_adjoint(sub, order, cdt, nd, steps, n_out):
    from paper_1408_7060_gb300 import abi

    f_c, dt, n0 = 150e6, cdt / C0, -4
    V, F, c = context(sub, order, dt, f_c)
    with c:
        r, wS = surface(c, V, F)
        rh, e1 = random_plane_waves(nd, 2)
        e2 = np.cross(rh, e1)
        rng = np.random.default_rng(5)
        I = rng.standard_normal((steps, c.ns)) + 1j * rng.standard_normal((steps, c.ns))
        G_in = rng.standard_normal((n_out, nd, 2)) + 1j * rng.standard_normal((n_out, nd, 2))
        got = abi.aim_farfield(c.handle, rh, e1, e2, I, n0, n_out)
        adj = abi.aim_farfield_adjoint(c.handle, rh, e1, e2, steps, n0, G_in)
        ref, radj = np.zeros_like(got), np.zeros_like(adj)
        wc = 2 * math.pi * f_c
        for d in range(nd):
            rr = r @ rh[d]
            ph = -MU0 / (4 * math.pi) * np.exp(1j * wc / C0 * rr)
            taps = {}
            for i in range(n_out):
                for l in range(steps):
                    s = n0 + i - (l + 1)
                    if s not in taps:
                        t = d_basis(s + rr / cdt, order, dt, wc) * ph
                        taps[s] = np.stack([(t * (wS @ e1[d])).sum(1), (t * (wS @ e2[d])).sum(1)], 1)
                    ref[i, d] += I[l] @ taps[s]
                    radj[l] += taps[s].conj() @ G_in[i, d]
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
    assert np.abs(adj - radj).max() <= 1e-12 * np.abs(radj).max()


@pytest.mark.parametrize("sub,f_mhz,nb,nf,nd", [(1, 100.0, 1, 1, 1), (2, 300.0, 5, 2, 33), (1, 2000.0, 2, 3, 300)])
def test_rcs(sub, f_mhz, nb, nf, nd):
    V, F, c = context(sub, 2, 0.8 / C0, 150e6)
    with c:
        r, wS = surface(c, V, F)
        rh, e1 = random_plane_waves(nd, 3)
        pol = e1 + 0.3 * rh  # the library projects it
        rng = np.random.default_rng(6)
        spec = rng.standard_normal((nf, nb, c.ns)) + 1j * rng.standard_normal((nf, nb, c.ns))
        freqs = f_mhz * 1e6 * (1.0 + 0.1 * np.arange(nf))
        got = c.rcs(freqs, spec, rh, pol)
    ref = np.zeros_like(got)
    for i, f in enumerate(freqs):
        w = 2 * math.pi * f
        for d in range(nd):
            v = (wS * np.exp(1j * w / C0 * (r @ rh[d]))[..., None]).sum(1)
            u = pol[d] - rh[d] * (rh[d] @ pol[d])
            ref[i, :, d] = 4 * math.pi * (w * MU0 / (4 * math.pi)) ** 2 * np.abs(spec[i] @ (v @ u)) ** 2
    assert np.abs(got - ref).max() < 1e-12 * ref.max()
