"""How the sums of aim_rcs round, against the same cubature in extended precision.

* The phase of a face is as exact as its vertices: on a sphere 64 m from the origin (phases
  of 400 radians at 300 MHz) and on finer spheres around the origin, the error is that of a
  few roundings per face, not of a phase rounded once for all 7 points of the face.
* A value does not depend on the other directions, frequencies and right-hand sides of the
  call: bitwise the same alone and among them.
* The work space stays within twice 64 MB and holds no room for right-hand sides that are not
  there, and a call of several passes over frequencies and directions gives the same values.

Bound of the first: a face's term (a u.(r - C) - u.b and the sums over its 7 points) passes
through about 16 roundings of relative size 2^-53, independent from face to face, and the
cross section doubles the amplitude's relative error, which leaves 16 x 2^-53 of the largest
value with a factor to spare (the roundings of hundreds of faces average).
"""
import math

import numpy as np
import pytest

from paper_1408_7060_gb300.inputs import icosphere, place_grid, random_plane_waves

pytestmark = pytest.mark.gpu

C0, MU0 = 299792458.0, 4e-7 * math.pi
LD = np.longdouble


def context(sub, shift=0.0, **kw):
    from paper_1408_7060_gb300 import AimContext

    V, F = icosphere(sub, 1.0)
    V = np.ascontiguousarray(V + shift * np.array([0.6, 0.64, 0.48]))
    h, origin = place_grid(V, 16, 0.15)
    return V, F, AimContext(V=V, F=F, grid_n=16, origin=origin, h=h, near_radius=-1.0, dt=0.8 / C0, f_c=150e6,
                            precision="c128", **kw)


def reference(c, V, F, f, spec, rh, pol):
    """The cross section of one spectrum in extended precision [nd] (k and the prefactor are
    the library's doubles: they are common factors)."""
    if np.finfo(LD).nmant < 63:
        pytest.skip("no extended precision on this machine")
    edge, tri, free = c.rwg_table()
    s15 = np.sqrt(LD(15))
    T = V.astype(LD)[F]
    ctr = T.sum(1) / 3
    pts, w = [ctr], [LD(9) / 40]
    for sg in (-1, 1):
        s = 1 - (6 + sg * s15) / 7
        for i in range(3):
            pts.append(ctr + s * (T[:, i] - ctr))
            w.append((155 + sg * s15) / 1200)
    q = np.stack(pts, 1)                                       # [nt][7][3]
    n = np.cross(T[:, 1] - T[:, 0], T[:, 2] - T[:, 0])
    area = np.sqrt((n * n).sum(1)) / 2
    d = V.astype(LD)[edge[:, 0]] - V.astype(LD)[edge[:, 1]]
    ln = np.sqrt((d * d).sum(1))
    k = 2.0 * math.pi * f / C0
    out = np.zeros(len(rh), LD)
    for i, (r, p) in enumerate(zip(rh.astype(LD), pol.astype(LD))):
        u = p - r * (r * p).sum()
        ph = LD(k) * (q * r).sum(2)
        wt = np.array(w)[None, :] * area[:, None]
        cs, sn = wt * np.cos(ph), wt * np.sin(ph)
        re = im = LD(0)
        for side, sign in ((0, 1), (1, -1)):
            t = tri[:, side]
            g = sign * ln[:, None] / (2 * area[t][:, None]) * ((q[t] - V.astype(LD)[free[:, side]][:, None]) * u).sum(2)
            a, b = (g * cs[t]).sum(1), (g * sn[t]).sum(1)
            x, y = spec.real.astype(LD), spec.imag.astype(LD)
            re += (x * a - y * b).sum()
            im += (x * b + y * a).sum()
        out[i] = re * re + im * im
    a = 2.0 * math.pi * f * MU0 / (4.0 * math.pi)
    return LD(4.0 * math.pi * a * a) * out


@pytest.mark.parametrize("sub,f,shift", [(1, 300e6, 64.0), (2, 300e6, 64.0), (3, 300e6, 0.0), (4, 600e6, 0.0)])
def test_phase_of_a_face(sub, f, shift):
    V, F, c = context(sub, shift)
    nd = 6
    with c:
        rh, pol = random_plane_waves(nd, 4)
        rng = np.random.default_rng(8)
        spec = rng.standard_normal(c.ns) + 1j * rng.standard_normal(c.ns)
        got = c.rcs([f], spec[None, None], rh, pol)[0, 0]
        ref = reference(c, V, F, f, spec, rh, pol)
    err = np.abs(got - ref) / ref.max()
    print(f"sub {sub} shift {shift}: {float(err.max()):.2e}")
    assert err.max() < 16 * 2.0 ** -53


@pytest.mark.parametrize("sub", [1, 3, 4])
def test_a_value_alone_and_among_others(sub):
    V, F, c = context(sub)
    nd, nb, freqs = 37, 6, 1e8 * np.array([1.0, 1.3, 2.0, 3.1, 4.4])
    with c:
        rh, pol = random_plane_waves(nd, 4)
        rng = np.random.default_rng(8)
        spec = rng.standard_normal((len(freqs), nb, c.ns)) + 1j * rng.standard_normal((len(freqs), nb, c.ns))
        got = c.rcs(freqs, spec, rh, pol)
        for f, b, d in ((0, 0, 0), (2, 3, 17), (4, 5, 36)):
            alone = c.rcs(freqs[f:f + 1], np.ascontiguousarray(spec[f:f + 1, b:b + 1]), rh[d:d + 1], pol[d:d + 1])
            assert alone[0, 0, 0] == got[f, b, d], (f, b, d)


def test_work_space_is_bounded():
    import torch

    from paper_1408_7060_gb300 import abi

    V, F, c = context(1)
    nd, nf = 9000, 500
    with c:
        rh, pol = random_plane_waves(nd, 4)
        freqs = np.linspace(1e8, 4e8, nf)
        spec = torch.randn(nf, 1, c.ns, dtype=torch.complex128, device="cuda")
        out = torch.empty(nf, 1, nd, dtype=torch.float64, device="cuda")
        before = abi.aim_get_info(c.handle)["device_bytes"]
        c.rcs(freqs, spec, rh, pol, out=out)
        assert abi.aim_get_info(c.handle)["device_bytes"] - before < 2 * (64 << 20) + (2 << 20)
        for f, d in ((0, 0), (nf - 1, nd - 1), (nf // 2, nd // 2)):
            alone = c.rcs(freqs[f:f + 1], spec[f:f + 1].contiguous(), rh[d:d + 1], pol[d:d + 1])
            assert float(alone[0, 0, 0]) == float(out[f, 0, d])
