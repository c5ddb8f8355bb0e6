"""The fused y/z passes on kx-major grids, at the sizes where their shapes change: every
padded length and z transform length, boxes that fill their transform and boxes much
thinner, one vector and odd batches, both precisions.  The products of the first and a
later delay and the delayed sum are compared with a plain FP64 evaluation (numpy FFTs on
the context's own stencil weights, kernel spectra and near values).

Tolerance: rounding.  The grid part is L^T F^-1 G F L x; each stage rounds relative to its
own size, so the error is at most a small multiple of eps max|G| |L_c x| |L_c| summed over
the components c (|L_c| bounded by the geometric mean of its largest row and column sums),
plus eps times the near part.  This bound does not shrink where the product is the small
difference of large parts (late delays inside the near zone).  The multiple is 8.
"""
import numpy as np
import pytest

from paper_1408_7060_gb300.inputs import icosphere, place_grid, plate_mesh

pytestmark = pytest.mark.gpu

F_C, BAND = 300e6, 0.3
# (mesh, z scale of a sphere or cells of a plate, grid, z transform length)
SIZES = [("sphere1", 1.0, 8, 16), ("sphere1", 0.2, 16, 16), ("sphere2", 1.0, 16, 32), ("plate", 9, 32, 16),
         ("sphere2", 0.3, 32, 32), ("sphere2", 1.0, 32, 64), ("plate", 14, 64, 16), ("sphere2", 0.15, 64, 32),
         ("sphere2", 0.4, 64, 64), ("sphere2", 1.0, 64, 128), ("plate", 21, 96, 16), ("sphere2", 0.5, 96, 128),
         ("sphere2", 1.0, 96, 192), ("plate", 30, 128, 16), ("sphere2", 0.4, 128, 128), ("sphere2", 0.72, 96, 144),
         ("sphere2", 0.53, 128, 144)]
# grids whose planes do not fit: separate y and z passes (and one whose z-spectral ring would
# take more than a quarter of the memory)
SEPARATE = [("sphere2", 0.7, 128, 192, "c64", 3, 3), ("sphere2", 1.0, 128, 256, "c64", 1, 1),
            ("sphere2", 1.0, 96, 192, "c64", 2, 160), ("sphere2", 0.72, 96, 144, "c128", 1, 1)]


def geometry(mesh, size, grid):
    if mesh == "plate":
        V, F = plate_mesh(0.1 * size, size)
    else:
        V, F = icosphere(int(mesh[-1]), 1.0)
        V = V * np.array([1.0, 1.0, size])
    h, origin = place_grid(V, grid)
    return V, F, h, origin


class Plain:
    def __init__(self, c):
        i = c.info
        L, lz = 2 * i["grid_n"], i["z_len"]
        a, self.lam = c.anterp()
        t = np.arange(64)
        x, y, z = a[:, :1] + (t & 3), a[:, 1:2] + ((t >> 2) & 3), a[:, 2:] - i["box_lo"][2] + (t >> 4)
        self.node, self.shape, self.c = (z * L + y) * L + x, (lz, L, L), c
        rowptr, self.col, self.val = c.near()
        self.row = np.repeat(np.arange(c.ns), np.diff(rowptr))

    def spectrum(self, m, kind):
        o = self.c.kernel_spectrum(m, kind)
        for d, n in enumerate(self.shape):
            o = np.take(o, np.minimum(np.arange(n), n - np.arange(n)), axis=d)
        return o * np.prod(self.shape)

    def product(self, m, x):
        """Z_m x and the rounding scale of its evaluation."""
        c, out = self.c, np.zeros(self.c.ns, complex)
        np.add.at(out, self.row, self.val[m] * x[self.col])
        scale = np.linalg.norm(out)
        G = [self.spectrum(m, 0), self.spectrum(m, 1)]
        for q in range(4):
            lam = np.abs(self.lam[:, q])
            cols = np.bincount(self.node.ravel(), lam.ravel())
            g = np.zeros(int(np.prod(self.shape)), complex)
            np.add.at(g, self.node.ravel(), (self.lam[:, q] * x[:, None]).ravel())
            scale += np.abs(G[q // 3]).max() * np.linalg.norm(g) * np.sqrt(lam.sum(1).max() * cols.max())
            g = np.fft.ifftn(np.fft.fftn(g.reshape(self.shape)) * G[q // 3]).ravel()
            out += (self.lam[:, q] * g[self.node]).sum(1)
        return out, scale


@pytest.mark.parametrize("mesh,size,grid,lz", SIZES)
@pytest.mark.parametrize("precision,nb", [("c64", 1), ("c64", 3), ("c128", 2)])
def test_products_and_sums(mesh, size, grid, lz, precision, nb):
    if grid > 64 and precision == "c128" and lz > 16:
        pytest.skip("the plain evaluation of the larger sizes runs once, in complex64")
    check(mesh, size, grid, lz, precision, nb, nb)


@pytest.mark.parametrize("mesh,size,grid,lz,precision,nb,batch_max", SEPARATE)
def test_separate_passes(mesh, size, grid, lz, precision, nb, batch_max):
    check(mesh, size, grid, lz, precision, nb, batch_max)


def check(mesh, size, grid, lz, precision, nb, batch_max):
    from paper_1408_7060_gb300 import AimContext

    V, F, h, origin = geometry(mesh, size, grid)
    rng = np.random.default_rng(3)
    with AimContext(V=V, F=F, grid_n=grid, origin=origin, h=h, near_radius=3 * h, dt=0.25 / (BAND * F_C), f_c=F_C,
                    precision=precision, batch_max=batch_max) as c:
        assert c.info["z_len"] == lz
        plain, ng = Plain(c), c.n_delays
        x = rng.standard_normal((ng, nb, c.ns)) + 1j * rng.standard_normal((ng, nb, c.ns))

        eps = 2.0 ** -53 if precision == "c128" else 2.0 ** -24
        b = nb - 1  # the last right-hand side of the batch
        for m in (0, ng):
            ref, scale = plain.product(m, x[0, b])
            assert np.linalg.norm(c.matvec(m, x[0])[b] - ref) < 8 * eps * scale, m
        refs = [plain.product(m, x[m - 1, b]) for m in range(1, ng + 1)]
        got = c.rhs(ng + 1, x)[b]
        assert np.linalg.norm(got - sum(r[0] for r in refs)) < 8 * eps * sum(r[1] for r in refs)
